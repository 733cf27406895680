// tensor.cuh -- LB-SMRT collide-and-stream on three-dimensional tensor-product velocity sets
// (Yan & Shan, arXiv 2401.11086, Sec. 4.2: the 3D products D3Q{d^3} of the 1D rules D1Qd-P1,
// D3Q729 = D1Q9-P1^3 of degree 11 and D3Q4913 = D1Q17-P1^3 of degree 19), batched 1D lines
// along x.
//
// A cell holds d^3 populations: too many for registers, so no pass ever holds them all. The
// projection (Eq. an) and the rebuild (Eq. fi) factor over the three axes because the
// abscissae, the weights and He_alpha(xi) = prod_k He_{alpha_k}(xi_k) all do:
//   a3  raw moments R_(j,k,l) = sum_{a,b,c} df_abc e_a^j e_b^k e_c^l, |(j,k,l)| <= N, summed
//       x first (one x-line of d populations at a time, +-e pairs folded), then y, then z;
//   a7  f'_abc = w_a w_b w_c sum_(j,k,l) P_(j,k,l) e_a^j e_b^k e_c^l, summed z first, then
//       y, then x, each x-line stored as soon as it is formed.
// With d = 9 and N = 5 that is about 4.6k multiply-adds each way instead of 41k for the
// dense d^3 x 56 products. Between the two, the moment-space steps a2, a4-a6 are those of the
// other velocity sets (core.cuh), acting on 56 coefficients in registers.
//
// Library order: population i = a + d b + d^2 c has velocity (e_a, e_b, e_c), where the 1D
// order is a = 0 rest, 2p+1 = +E_p, 2p+2 = -E_p. The caller's order is arbitrary: its plane
// index for every library population sits in a table that each block copies to shared memory.
// Ghost populations (end states beyond a fixed x end) are kept in library order.
#pragma once


#include "kernels.cuh"
#include "lane_kernels.cuh"

namespace smrt {

// D1Q9-P1 (Table 3, d = 9, degree 11): abscissae c {0, +-1, +-2, +-3, +-5}.
struct D1Q9P1 {
    static constexpr int Q1 = 9;
    static constexpr int NP1 = 4;
    static constexpr int DEGREE = 11;
    static constexpr double C_GUESS = 0.678;  // start of the scale search in the host solver
    static constexpr SMRT_HD int E(int p) { return p < 3 ? p + 1 : 5; }
};

// D1Q17-P1 (Table 3, d = 17, degree 19): abscissae c {0, +-1, ..., +-7, +-9}.
struct D1Q17P1 {
    static constexpr int Q1 = 17;
    static constexpr int NP1 = 8;
    static constexpr int DEGREE = 19;
    static constexpr double C_GUESS = 0.5639;
    static constexpr SMRT_HD int E(int p) { return p < 7 ? p + 1 : 9; }
};

template <class L1>
constexpr SMRT_HD int e1(int a) {
    return a == 0 ? 0 : ((a & 1) ? L1::E((a - 1) / 2) : -L1::E((a - 1) / 2));
}

constexpr int kMaxQ1 = 17;

// Basis of the x-passes: instead of the powers e^j, polynomials of the same degree and parity with as
// many zeros on the abscissae 0, +-1, +-2 as their degree allows,
//   1, e, e^2, e (e^2 - 1) / 6, e^2 (e^2 - 1) / 12, e (e^2 - 1) (e^2 - 4) / 120,
// integers at every abscissa, 1 at the first one where they do not vanish. A row of D1Q9-P1 then
// takes 15 multiply-adds instead of 24 in the projection and 12 instead of 20 in the rebuild
// (39 instead of 48, and 28 instead of 40, on D1Q17-P1); the change to and from the powers acts once per cell on the
// 56 moments (x_to_powers, x_from_powers).
constexpr int xbasis(int j, int e) {
    const int q = e * e;
    return j == 0   ? 1
           : j == 1 ? e
           : j == 2 ? q
           : j == 3 ? e * (q - 1) / 6
           : j == 4 ? q * (q - 1) / 12
                    : e * (q - 1) * (q - 4) / 120;
}

template <class T>
struct TPArgs {
    const T *__restrict__ fin;
    T *__restrict__ fout;
    const InstanceInfo *__restrict__ inst;
    const int2 *__restrict__ tiles;    // (instance, first x) per block
    const T *__restrict__ ghosts;      // [instance][2][Q], library order
    unsigned *health;
    const int *__restrict__ plane_idx; // caller plane of each library population
    long long stride;                  // elements per population plane
    double cd;                         // lattice scale c
    double w1[kMaxQ1];                 // 1D weights, library order
    unsigned step;
    int tma;                           // 1: the kernel's tensor maps describe fin and fout
    int ident;                         // 1: library population i is caller plane i
};

// Tensor maps of the two states for the block-staged kernels: a 2D view [plane][stride] of a
// state (library order = caller order), box of kSeg elements x d planes (one x-row group).
struct TPMaps {
    CUtensorMap src;  // of TPArgs::fin
    CUtensorMap dst;  // of TPArgs::fout
};

// Shared-memory tables of one block: caller planes (Planes; the block-staged step reads them
// from global memory, and only when the caller's order is not the library's), the 1D abscissae
// (integers, as T) and the 1D weights (as T).
template <class L1, class T, bool Planes = true>
struct TPTables {
    static constexpr int Q = L1::Q1 * L1::Q1 * L1::Q1;
    static constexpr int kPow = 6;  // powers e^0 .. e^5 (N <= 5)
    int plane[Planes ? Q : 1];
    T e[L1::Q1];
    T w[L1::Q1];
    T pw[L1::Q1][kPow];  // e_a^k: the y and z passes read them instead of forming them per cell
};

template <class L1, class T, class U, bool Planes>
SMRT_D void tp_load_tables(const TPArgs<T> &a, TPTables<L1, U, Planes> &s) {
    if constexpr (Planes)
        for (int i = threadIdx.x; i < TPTables<L1, U>::Q; i += blockDim.x) s.plane[i] = a.plane_idx[i];
    if (threadIdx.x < L1::Q1) {
        const U ea = U(e1<L1>(threadIdx.x));
        s.e[threadIdx.x] = ea;
        s.w[threadIdx.x] = U(a.w1[threadIdx.x]);
        U p = U(1);
        for (int k = 0; k < TPTables<L1, U>::kPow; ++k, p *= ea) s.pw[threadIdx.x][k] = p;
    }
    __syncthreads();
}

// The step's tables: also the weights w_a w_b w_c by the classes (rest, then each pair) of c, b, a,
// rounded once and read per x-row. One row per unordered pair (b, c): a row per ordered pair took
// 5.8 KB on D1Q17-P1 in double, and the third two-warp block no longer fitted an SM (24 shocks of
// 1000 cells, N = 5: 3.32 ms per step with two blocks, 2.45 with three).
template <class L1, class T, bool Planes = true>
struct TPStepTables : TPTables<L1, T, Planes> {
    static constexpr int K = L1::NP1 + 1;
    T w3[K * (K + 1) / 2][K];
    SMRT_HD static constexpr int row(int b, int c) { return b > c ? b * (b + 1) / 2 + c : c * (c + 1) / 2 + b; }
};

template <class L1, class T, bool Planes>
SMRT_D void tp_load_step_tables(const TPArgs<T> &a, TPStepTables<L1, T, Planes> &s) {
    constexpr int K = TPStepTables<L1, T, Planes>::K;
    for (int i = threadIdx.x; i < K * K * K; i += blockDim.x) {
        const int c = i / (K * K), b = i / K % K, q = i % K;  // class p > 0: abscissae 2 p - 1, 2 p
        if (b <= c)
            s.w3[s.row(b, c)][q] = T(a.w1[c ? 2 * c - 1 : 0] * a.w1[b ? 2 * b - 1 : 0] * a.w1[q ? 2 * q - 1 : 0]);
    }
    tp_load_tables<L1>(a, static_cast<TPTables<L1, T, Planes> &>(s));  // ends with __syncthreads
}

// Two floats in one 64-bit register pair: one packed instruction (add / multiply / fused
// multiply-add, each lane rounded as the scalar one) works on both.
struct F2 {
    unsigned long long v;
    F2() = default;
    SMRT_D F2(float a, float b) { asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b)); }
    SMRT_D F2(float a) : F2(a, a) {}
    SMRT_D F2(double a) : F2(float(a), float(a)) {}
    SMRT_D F2(int a) : F2(float(a), float(a)) {}
    SMRT_D float lo() const { return __uint_as_float(static_cast<unsigned>(v)); }
    SMRT_D float hi() const { return __uint_as_float(static_cast<unsigned>(v >> 32)); }
    // friends: found for F2 arguments only (fma of floats and doubles stays the global one)
    SMRT_D friend F2 operator+(F2 a, F2 b) {
        F2 r;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
        return r;
    }
    SMRT_D friend F2 operator*(F2 a, F2 b) {
        F2 r;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
        return r;
    }
    SMRT_D friend F2 fma(F2 a, F2 b, F2 c) {
        F2 r;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
        return r;
    }
    SMRT_D friend F2 operator-(F2 a, F2 b) { return fma(F2(-1.f), b, a); }
};

template <class L1, int N, class T>
struct TPCell {
    static constexpr int Q1 = L1::Q1;
    static constexpr int NP1 = L1::NP1;
    static constexpr int M = nmom(N);

    // R_(j,k,l) from the basis of the x-passes to powers of e_x ...
    template <class U>
    SMRT_D static void x_to_powers(U (&R)[M]) {
        for_j<5>([&](auto K, auto L) {
            constexpr int k = decltype(K)::value, l = decltype(L)::value;
            R[mi_pos(5, k, l)] = fma(U(120), R[mi_pos(5, k, l)], fma(U(30), R[mi_pos(3, k, l)], R[mi_pos(1, k, l)]));
        });
        for_j<4>([&](auto K, auto L) {
            constexpr int k = decltype(K)::value, l = decltype(L)::value;
            R[mi_pos(4, k, l)] = fma(U(12), R[mi_pos(4, k, l)], R[mi_pos(2, k, l)]);
        });
        for_j<3>([&](auto K, auto L) {
            constexpr int k = decltype(K)::value, l = decltype(L)::value;
            R[mi_pos(3, k, l)] = fma(U(6), R[mi_pos(3, k, l)], R[mi_pos(1, k, l)]);
        });
    }
    // ... and the coefficients of powers of e_x to those of the basis
    template <class U>
    SMRT_D static void x_from_powers(U (&P)[M]) {
        for_j<3>([&](auto K, auto L) {
            constexpr int k = decltype(K)::value, l = decltype(L)::value;
            P[mi_pos(1, k, l)] += P[mi_pos(3, k, l)];
            P[mi_pos(3, k, l)] *= U(6);
        });
        for_j<4>([&](auto K, auto L) {
            constexpr int k = decltype(K)::value, l = decltype(L)::value;
            P[mi_pos(2, k, l)] += P[mi_pos(4, k, l)];
            P[mi_pos(4, k, l)] *= U(12);
        });
        for_j<5>([&](auto K, auto L) {
            constexpr int k = decltype(K)::value, l = decltype(L)::value;
            P[mi_pos(1, k, l)] += P[mi_pos(5, k, l)];
            P[mi_pos(3, k, l)] = fma(U(30), P[mi_pos(5, k, l)], P[mi_pos(3, k, l)]);
            P[mi_pos(5, k, l)] *= U(120);
        });
    }
    // every (k, l) with j + k + l <= N (none when j > N)
    template <int j, class F>
    SMRT_HD static void for_j(F &&f) {
        static_for<(N >= j ? N - j + 1 : 0)>([&](auto K) {
            constexpr int k = decltype(K)::value;
            static_for<N - j - k + 1>([&](auto L) { f(ic<k>{}, L); });
        });
    }

    // a1 + a3: raw moments of the pulled populations; pop(i, ic<a>) returns population i
    // (library index) whose x-velocity index is a.
    template <class Pop>
    SMRT_D static void project(Pop &&pop, const T *s_e, T (&R)[M]) {
        static_for<M>([&](auto G) { R[decltype(G)::value] = T(0); });
#pragma unroll 1
        for (int cz = 0; cz < Q1; ++cz) {
            T h[N + 1][N + 1];
            static_for<N + 1>([&](auto J) {
                static_for<N + 1 - decltype(J)::value>([&](auto K) { h[decltype(J)::value][decltype(K)::value] = T(0); });
            });
            const int i0 = cz * Q1 * Q1;
            {  // b = rest: only k = 0
                T g[N + 1];
                xrow([&](auto A) -> T { return pop(i0 + decltype(A)::value, A); }, g);
                static_for<N + 1>([&](auto J) { h[decltype(J)::value][0] += g[decltype(J)::value]; });
            }
            static_for<NP1>([&](auto P) {
                constexpr int p = decltype(P)::value;
                T gp[N + 1], gm[N + 1];
                xrow([&](auto A) -> T { return pop(i0 + Q1 * (2 * p + 1) + decltype(A)::value, A); }, gp);
                xrow([&](auto A) -> T { return pop(i0 + Q1 * (2 * p + 2) + decltype(A)::value, A); }, gm);
                static_for<N + 1>([&](auto J) {
                    constexpr int j = decltype(J)::value;
                    const T s = gp[j] + gm[j], d = gp[j] - gm[j];
                    static_for<N + 1 - j>([&](auto K) {
                        constexpr int k = decltype(K)::value;
                        constexpr double ek = double(ipow(L1::E(p), k));
                        if constexpr (k == 0)
                            h[j][0] += s;
                        else if constexpr (k & 1)
                            h[j][k] = fma(T(ek), d, h[j][k]);
                        else
                            h[j][k] = fma(T(ek), s, h[j][k]);
                    });
                });
            });
            const T ec = s_e[cz];
            T pw[N + 1];
            pw[0] = T(1);
            static_for<N>([&](auto L) { pw[decltype(L)::value + 1] = pw[decltype(L)::value] * ec; });
            static_for<M>([&](auto G) {
                constexpr int g = decltype(G)::value;
                constexpr int j = mi_comp(g, 0), k = mi_comp(g, 1), l = mi_comp(g, 2);
                if constexpr (l == 0)
                    R[g] += h[j][k];
                else
                    R[g] = fma(pw[l], h[j][k], R[g]);
            });
        }
        x_to_powers(R);
    }

    // Pieces of the same sums for a pipeline that sees one +-e_b pair of x-rows at a time.
    // g_j = sum_a f_a b_j(e_a) over one x-row, b_j the basis above; row(ic<a>) returns the population
    // with x-index a.
    template <class Row>
    SMRT_D static void xrow(const Row &row, T (&g)[N + 1]) {
        const T f0 = row(ic<0>{});
        T S[NP1], D[NP1];
        static_for<NP1>([&](auto P) {
            constexpr int p = decltype(P)::value;
            const T fp = row(ic<2 * p + 1>{});
            const T fm = row(ic<2 * p + 2>{});
            S[p] = fp + fm;
            D[p] = fp - fm;
        });
        static_for<N + 1>([&](auto J) {
            constexpr int j = decltype(J)::value;
            T acc = f0;  // j > 0: replaced by the first term, whose coefficient is 1
            static_for<NP1>([&](auto P) {
                constexpr int p = decltype(P)::value;
                constexpr int v = xbasis(j, L1::E(p)), before = p > 0 ? xbasis(j, L1::E(p > 0 ? p - 1 : 0)) : 0;
                const T x = (j & 1) ? D[p] : S[p];
                if constexpr (j == 0)
                    acc = acc + x;
                else if constexpr (v != 0 && before == 0)
                    acc = x;
                else if constexpr (v != 0)
                    acc = fma(T(v), x, acc);
                static_assert(j == 0 || v == 0 || before != 0 || v == 1, "1 at the first abscissa where it does not vanish");
            });
            g[j] = acc;
        });
    }
    // h_(j,k) += sum_b g_(b)j e_b^k for the rest row (e_b = 0) ...
    SMRT_D static void yrest(const T (&g)[N + 1], T (&h)[N + 1][N + 1]) {
        static_for<N + 1>([&](auto J) { h[decltype(J)::value][0] += g[decltype(J)::value]; });
    }
    // ... and for the rows +e_b (gp) and -e_b (gm)
    SMRT_D static void ypair(const T (&gp)[N + 1], const T (&gm)[N + 1], T eb, T (&h)[N + 1][N + 1]) {
        T pw[N + 1];
        pw[0] = T(1);
        static_for<N>([&](auto K) { pw[decltype(K)::value + 1] = pw[decltype(K)::value] * eb; });
        ypair_pw(gp, gm, pw, h);
    }
    // ... with the powers e_b^k given (pw[k], k <= N, e.g. a shared-memory table row)
    template <class PW>
    SMRT_D static void ypair_pw(const T (&gp)[N + 1], const T (&gm)[N + 1], const PW &pw, T (&h)[N + 1][N + 1]) {
        static_for<N + 1>([&](auto J) {
            constexpr int j = decltype(J)::value;
            const T s = gp[j] + gm[j], d = gp[j] - gm[j];
            h[j][0] += s;
            static_for<N - j>([&](auto K) {
                constexpr int k = decltype(K)::value + 1;
                h[j][k] = fma(pw[k], (k & 1) ? d : s, h[j][k]);
            });
        });
    }
    // R_(j,k,l) += e_c^l h_(j,k) at the end of z-plane c; h is cleared for the next one
    SMRT_D static void zfold(T (&h)[N + 1][N + 1], T ec, T (&R)[M]) {
        T pw[N + 1];
        pw[0] = T(1);
        static_for<N>([&](auto L) { pw[decltype(L)::value + 1] = pw[decltype(L)::value] * ec; });
        zfold_pw(h, pw, R);
    }
    template <class PW>
    SMRT_D static void zfold_pw(T (&h)[N + 1][N + 1], const PW &pw, T (&R)[M]) {
        static_for<M>([&](auto G) {
            constexpr int g = decltype(G)::value;
            constexpr int j = mi_comp(g, 0), k = mi_comp(g, 1), l = mi_comp(g, 2);
            if constexpr (l == 0)
                R[g] += h[j][k];
            else
                R[g] = fma(pw[l], h[j][k], R[g]);
        });
        static_for<N + 1>([&](auto J) {
            static_for<N + 1 - decltype(J)::value>([&](auto K) { h[decltype(J)::value][decltype(K)::value] = T(0); });
        });
    }
    // Rebuild side: Pc_(j,k) = sum_l P_(j,k,l) e_c^l for z-plane c (pw[l] = e_c^l) ...
    template <class U, class PW>
    SMRT_D static void zplane_pw(const U (&P)[M], const PW &pw, U (&Pc)[N + 1][N + 1]) {
        static_for<N + 1>([&](auto J) {
            constexpr int j = decltype(J)::value;
            static_for<N + 1 - j>([&](auto K) {
                constexpr int k = decltype(K)::value;
                U acc = P[mi_pos(j, k, 0)];
                static_for<N - j - k>([&](auto L) {
                    constexpr int l = decltype(L)::value + 1;
                    acc = fma(pw[l], P[mi_pos(j, k, l)], acc);
                });
                Pc[j][k] = acc;
            });
        });
    }
    // ... and the x-row coefficients Pb_j = sum_k Pc_(j,k) (+-e_b)^k of the rows +e_b, -e_b
    template <class U, class PW>
    SMRT_D static void yrows_pw(const U (&Pc)[N + 1][N + 1], const PW &pw, U (&Pp)[N + 1], U (&Pm)[N + 1]) {
        static_for<N + 1>([&](auto J) {
            constexpr int j = decltype(J)::value;
            U ev = Pc[j][0], od = U(0);
            static_for<N - j>([&](auto K) {
                constexpr int k = decltype(K)::value + 1;
                if constexpr (k == 1)
                    od = pw[k] * Pc[j][k];
                else if constexpr (k & 1)
                    od = fma(pw[k], Pc[j][k], od);
                else
                    ev = fma(pw[k], Pc[j][k], ev);
            });
            Pp[j] = ev + od;
            Pm[j] = ev - od;
        });
    }

    SMRT_D static void relax_es(T (&v)[M], T rho, T A, T B, T b) { relax_es_divided<N, T>(v, rho, A, B, b); }

    // a2, a4-a6 on the raw moments: R (in) -> rebuild coefficients P (out, same slots) with
    // f'_i = w_i sum_gamma P_gamma e_i^gamma. model 1: ES-BGK with parameter es_b, else SMRT.
    // Returns false when rho or theta is not positive.
    SMRT_D static bool collide_moments(T (&R)[M], T c, const T *tauA, const T *tauB, int model = 0,
                                       T es_b = T(0)) {
        T cp[N + 1];
        cp[0] = T(1);
        static_for<N>([&](auto J) { cp[decltype(J)::value + 1] = cp[decltype(J)::value] * c; });
        T Rc[M];
        static_for<M>([&](auto G) {
            constexpr int g = decltype(G)::value;
            Rc[g] = R[g] * cp[mi_order(g)];
        });
        // a2: rho - 1 = Rc_0, rho u = Rc_1, E - 3 = tr Rc_2 (deviations from w_i)
        const T rhom1 = Rc[0];
        const T rho = T(1) + rhom1;
        const T ir = rcp(rho);
        const T u[3] = {Rc[mi_pos(1, 0, 0)] * ir, Rc[mi_pos(0, 1, 0)] * ir, Rc[mi_pos(0, 0, 1)] * ir};
        const T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        const T em3 = Rc[mi_pos(2, 0, 0)] + Rc[mi_pos(0, 2, 0)] + Rc[mi_pos(0, 0, 2)];
        const T thm1 = (em3 - T(3) * rhom1 - rho * uu) * ir * T(1.0 / 3.0);
        const T theta = T(1) + thm1;
        const bool ok = (rho > T(0)) && (theta > T(0));
        // a3 (end): ta_alpha = a_alpha / alpha! = sum_gamma hdiv(alpha, gamma) Rc_gamma
        T v[M];
        static_for<M>([&](auto A) {
            constexpr int al = decltype(A)::value;
            T acc = T(0);
            static_for<M>([&](auto G) {
                constexpr int g = decltype(G)::value;
                constexpr double h = hdiv(al, g);
                if constexpr (h != 0.0) acc = fma(T(h), Rc[g], acc);
            });
            v[al] = acc;
        });
        v[0] = rho;
        to_local_divided<N, T>(v, u, theta, thm1);
        // a5
        if (model == 1) {
            relax_es(v, rho, tauA[0], tauB[0], es_b);
        } else {
            T s[ntau(N)];
            static_for<ntau(N)>([&](auto K) {
                constexpr int k = decltype(K)::value;
                s[k] = T(1) - rcp_tau<T>(tauA[k], tauB[k], rho);
            });
            static_for<N - 1>([&](auto Nn) { relax_order<N, decltype(Nn)::value + 2, T>(v, s); });
        }
        // a6
        const T sq = theta * rsq(theta);
        T sp[N + 1];
        sp[0] = T(1);
        static_for<N>([&](auto J) { sp[decltype(J)::value + 1] = sp[decltype(J)::value] * sq; });
        static_for<M>([&](auto A) {
            constexpr int p = decltype(A)::value;
            if constexpr (mi_order(p) == 0)
                v[p] = rho;
            else if constexpr (mi_order(p) == 1)
                v[p] = T(0);
            else
                v[p] *= sp[mi_order(p)];
        });
        T G[3][N + 1];
        static_for<3>([&](auto K) {
            constexpr int k = decltype(K)::value;
            maxwell_divided<N, T>(G[k], u[k], thm1);
        });
        binomial_divided<N, T>(v, G);
        v[0] = rhom1;  // deviation from the coefficients of w_i
        to_rebuild(v, c, R);
        return ok;
    }

    // P_gamma = c^|gamma| sum_alpha hfull(alpha, gamma) ta_alpha (the monomial form of Eq. fi)
    template <class U>
    SMRT_D static void to_rebuild(const U (&ta)[M], U c, U (&P)[M]) {
        U cp[N + 1];
        cp[0] = U(1);
        static_for<N>([&](auto J) { cp[decltype(J)::value + 1] = cp[decltype(J)::value] * c; });
        static_for<M>([&](auto G) {
            constexpr int g = decltype(G)::value;
            U acc = U(0);
            static_for<M>([&](auto A) {
                constexpr int al = decltype(A)::value;
                constexpr double h = hfull(al, g);
                if constexpr (h != 0.0) acc = fma(U(h), ta[al], acc);
            });
            P[g] = acc * cp[mi_order(g)];
        });
    }

    // One x-row of the rebuild from its coefficients Pb in the basis of the x-passes:
    // f'_(a,b,c) = w (ev +- E od), od the odd part over E; w: w_a w_b w_c by the class of a.
    template <class U, class W, class Put>
    SMRT_D static void emit_x(const U (&Pb)[N + 1], const W &w, int i0, Put &put) {
        put(i0, U(w[0]) * Pb[0]);
        static_for<NP1>([&](auto Q) {
            constexpr int q = decltype(Q)::value, E = L1::E(q);
            U ev = Pb[0], od = Pb[1];
            static_for<N - 1>([&](auto J) {
                constexpr int j = decltype(J)::value + 2, v = xbasis(j, E);
                if constexpr (v != 0 && (j & 1))
                    od = fma(U(double(v) / E), Pb[j], od);
                else if constexpr (v == 1)
                    ev = ev + Pb[j];
                else if constexpr (v != 0)
                    ev = fma(U(v), Pb[j], ev);
            });
            const U wq = w[q + 1];
            put(i0 + 2 * q + 1, wq * fma(U(E), od, ev));
            put(i0 + 2 * q + 2, wq * fma(U(-E), od, ev));
        });
    }

    // a7: every population from the rebuild coefficients P (in powers of e; left in the basis of the
    // x-passes); put(i, value) receives population i (library index). s_e, s_w: 1D abscissae and
    // weights in U.
    template <class U, class Put>
    SMRT_D static void rebuild(U (&P)[M], const U *s_e, const U *s_w, Put &&put) {
        x_from_powers(P);
        U wx[NP1 + 1];
        wx[0] = s_w[0];
        static_for<NP1>([&](auto Pp) { wx[decltype(Pp)::value + 1] = s_w[2 * decltype(Pp)::value + 1]; });
#pragma unroll 1
        for (int cz = 0; cz < Q1; ++cz) {
            const U ec = s_e[cz], wc = s_w[cz];
            U pw[N + 1];
            pw[0] = U(1);
            static_for<N>([&](auto L) { pw[decltype(L)::value + 1] = pw[decltype(L)::value] * ec; });
            U Pc[N + 1][N + 1], w[NP1 + 1];
            zplane_pw(P, pw, Pc);
            const int i0 = cz * Q1 * Q1;
            {  // b = rest
                U Pb[N + 1];
                static_for<N + 1>([&](auto J) { Pb[decltype(J)::value] = Pc[decltype(J)::value][0]; });
                static_for<NP1 + 1>([&](auto Q) { w[decltype(Q)::value] = wc * wx[0] * wx[decltype(Q)::value]; });
                emit_x(Pb, w, i0, put);
            }
            static_for<NP1>([&](auto Pp) {
                constexpr int p = decltype(Pp)::value;
                U py[N + 1], Pr[N + 1], Pm[N + 1];
                static_for<N + 1>([&](auto K) { py[decltype(K)::value] = U(ipow(L1::E(p), decltype(K)::value)); });
                yrows_pw(Pc, py, Pr, Pm);
                static_for<NP1 + 1>([&](auto Q) { w[decltype(Q)::value] = wc * wx[p + 1] * wx[decltype(Q)::value]; });
                emit_x(Pr, w, i0 + Q1 * (2 * p + 1), put);
                emit_x(Pm, w, i0 + Q1 * (2 * p + 2), put);
            });
        }
    }

    // Order-N equilibrium of (rho, u, theta) as deviations from w_i: rebuild coefficients in U.
    template <class U>
    SMRT_D static void equilibrium(U rho, const U (&u)[3], U theta, U c, U (&P)[M]) {
        U G[3][N + 1];
        static_for<3>([&](auto K) {
            constexpr int k = decltype(K)::value;
            maxwell_divided<N, U>(G[k], u[k], theta - U(1));
        });
        U ta[M];
        static_for<M>([&](auto A) {
            constexpr int p = decltype(A)::value;
            ta[p] = rho * G[0][mi_comp(p, 0)] * G[1][mi_comp(p, 1)] * G[2][mi_comp(p, 2)];
        });
        ta[0] = rho - U(1);
        to_rebuild<U>(ta, c, P);
    }
};

// One plain arrival on mbarrier b (a warp's release of a stage buffer).
SMRT_D void mbar_arrive(unsigned long long *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(b)) : "memory");
}
// One element global -> shared by an asynchronous copy (4 or 8 bytes, element-aligned) ...
template <class T>
SMRT_D void cp_async_elem(T *dst, const T *src) {
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "4- or 8-byte elements");
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst)), "l"(src), "n"(int(sizeof(T)))
                 : "memory");
}
// ... and the phase of mbarrier b waits for every such copy this thread has issued (the
// barrier's pending count is raised now and lowered when they complete).
SMRT_D void cp_async_mbar_arrive(unsigned long long *b) {
    asm volatile("cp.async.mbarrier.arrive.shared::cta.b64 [%0];" ::"r"(smem_addr(b)) : "memory");
}

// ------------------------------------------------------------------ block-staged line tile
// A block of W warps owns a tile of 32 W consecutive cells of one line (warp w takes cells
// 32 w .. 32 w + 31, one per lane) and one copy pipeline. The step's d^3 pulls per cell reach
// shared memory by stage: stage st covers z-plane c = st / (NP1 + 1) and, within it, either the
// rest x-row (e_b = 0, d planes) or the pair of x-rows +e_b, -e_b (2 d planes). Each plane
// arrives as one contiguous x-segment [x0 - k - E_max, x0 + 32 W - 1 - k + E_max] (every pull of
// the tile, rounded out to 16 bytes) that all the block's warps read, so a halo of 2 E_max is
// loaded once per 32 W cells and each copied row is 32 W cells long. kStages fills are in
// flight: each buffer has a "full" mbarrier (the copy's bytes) and an "empty" one (one arrival
// per warp that is done with the buffer), which warp 0 waits on before refilling it. No
// block-wide barrier is taken inside a tile; the warps drift up to kStages stages apart.
// (Measured on 512 Table 3 shocks, D3Q729 float, 128-cell tiles: 0.248 ms per step; five
// stages 0.271 ms; refills issued by whichever warp releases a buffer last, counted by shared
// atomics, 0.259 ms; one warp per tile, 0.287 ms.)
template <class L1, class T, int W>
struct TPBlockStage {
    static constexpr int kW = 32 * W;                   // cells per block tile
    static constexpr int kStages = 3;                   // fills in flight per block
    static constexpr int kAlign = 16 / int(sizeof(T));  // elements per 16 bytes
    static constexpr int kEmax = L1::E(L1::NP1 - 1);    // largest |e| of the 1D rule
    static constexpr int kSeg = kW + ((2 * kEmax + kAlign - 1) + kAlign - 1) / kAlign * kAlign;
    static_assert(kSeg <= 256, "a tensor-map box spans at most 256 elements");
    // a stage buffer holds two groups of d rows (the +e_b and -e_b x-rows), each group starting
    // 128-byte aligned so that one tensor-map box fills it, and after its rows the end-state
    // populations of its planes, [left, right][d], for the pulls from beyond a line's fixed ends
    static constexpr int kEnds = L1::Q1 * kSeg;
    static constexpr int kGrp = int(((kEnds + 2 * L1::Q1) * sizeof(T) + 127) / 128 * 128 / sizeof(T));
    static constexpr int kStage = 2 * kGrp;             // elements per stage buffer
    static constexpr int kPerZ = L1::NP1 + 1;           // stages per z-plane
    static constexpr int kTotal = L1::Q1 * kPerZ;       // stages per step
    static_assert(kTotal % kStages == 0, "each tile starts the buffers' cycle at buffer 0");
    static_assert(kStages * 16 <= 128, "the full and empty mbarriers fit the 128-byte head");
    static constexpr size_t kBytes = 128 + size_t(kStages) * kStage * sizeof(T);  // mbarriers, buffers
};

// An SM's shared memory: 228 KB, of which each block takes 1 KB beside its own.
constexpr size_t kSharedPerSM = 228 * 1024, kSharedPerBlock = 1024;
// The double D1Q17-P1 step, bound by the FP64 pipe that an SM's warps share, keeps three blocks of
// its two-warp tiles resident (128: the kernels' own scalars).
static_assert(3 * (TPBlockStage<D1Q17P1, double, 2>::kBytes + sizeof(TPStepTables<D1Q17P1, double, false>) + 128 +
                   kSharedPerBlock) <= kSharedPerSM,
              "three blocks fit an SM");

// ------------------------------------------------------------------ x-row sums on tensor cores
// The x-row sums of one stage, g_j = sum_a f_a e_a^j for each of the warp's 32 cells and the
// stage's one or two x-rows, as one warp-wide matrix product: rows (x-row, cell), columns
// j = 0..7 (those above N are zero), inner index a = 1 .. d - 1 in k-steps of 8; the rest
// velocity (e_0 = 0) adds to g_0 only and seeds the accumulator. mma.sync m16n8k8 with TF32
// operands and FP32 accumulation; single-precision accuracy from the operand split of Ootomo &
// Yokota (2022, "Recovering single precision accuracy from Tensor Cores while surpassing the
// FP32 theoretical peak performance"): f = f_hi + f_lo with f_hi = f rounded to TF32 and f_lo
// the remainder rounded to TF32 (each rounding within 2^-11 relative), e^j = E_hi + E_lo
// likewise and exactly (e^j <= 9^5 has at most 16 significant bits, E_lo at most 5), and
// g = f_lo E_hi + f_hi E_lo + f_hi E_hi; the dropped f_lo E_lo and the rounding of f_lo are
// each below 2^-22 of |f| e^j.
// m16n8k8 TF32 fragments, lane = 4 r + q: A rows r and r + 8, columns q and q + 4; B rows
// (inner index) q and q + 4, column r; C rows r and r + 8, columns 2q and 2q + 1.
template <class L1, int N>
struct TPTensorRows {
    static constexpr int KS = (L1::Q1 - 1) / 8;  // k-steps over a = 1 .. d - 1
    static_assert((L1::Q1 - 1) % 8 == 0 && N + 1 <= 8, "k-steps of 8 velocities, j <= 7");
    static constexpr int kPitch = 10;            // floats per (x-row, cell) row of the scratch
    unsigned bhi[KS][2], blo[KS][2];             // B fragments, e_a^j split in two
    int off[KS][2];                              // a SEG - e_a for the lane's two columns
    int r, q;

    SMRT_D static unsigned tf32(float x) {
        unsigned u;
        asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
        return u;
    }
    SMRT_D static void mma(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
        asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
            "{%8, %9}, {%0, %1, %2, %3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    }

    // seg: elements per staged row
    SMRT_D void init(int lane, int seg) {
        r = lane >> 2;
        q = lane & 3;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int av = 8 * ks + q + 4 * h + 1;
                int e = 0;
                static_for<L1::Q1>([&](auto A) {
                    if (decltype(A)::value == av) e = e1<L1>(decltype(A)::value);
                });
                off[ks][h] = av * seg - e;
                float pw = r <= N ? 1.f : 0.f;  // e^r, exact in float
                for (int j = 0; j < r; ++j) pw *= float(e);
                const unsigned hi = tf32(pw);
                bhi[ks][h] = hi;
                blo[ks][h] = tf32(pw - __uint_as_float(hi));
            }
    }

    // g[x][j], x < NR, for the lane's cell: the pull of x-row x by velocity a of cell c sits at
    // bs[x grp + a SEG + tb0 + c - e_a]. Every lane calls it. The first NR 32 kPitch floats of bs
    // serve as scratch to hand each cell its row sums, so bs is overwritten.
    template <int NR>
    SMRT_D void rows(float *bs, int grp, int tb0, int lane, float (&g)[NR][N + 1]) const {
        float acc[NR][2][4];
#pragma unroll
        for (int x = 0; x < NR; ++x)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const float *p = bs + x * grp + tb0 + 16 * mt + r;
                float(&d)[4] = acc[x][mt];
                d[0] = q == 0 ? p[0] : 0.f;  // the rest velocity: column j = 0
                d[1] = 0.f;
                d[2] = q == 0 ? p[8] : 0.f;
                d[3] = 0.f;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
                    const float v[4] = {p[off[ks][0]], p[off[ks][0] + 8], p[off[ks][1]], p[off[ks][1] + 8]};
                    unsigned ahi[4], alo[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        ahi[i] = tf32(v[i]);
                        alo[i] = tf32(v[i] - __uint_as_float(ahi[i]));
                    }
                    mma(d, alo, bhi[ks][0], bhi[ks][1]);
                    mma(d, ahi, blo[ks][0], blo[ks][1]);
                    mma(d, ahi, bhi[ks][0], bhi[ks][1]);
                }
            }
        __syncwarp();  // every lane holds its operands: the buffer is free
        if (2 * q <= N) {
#pragma unroll
            for (int x = 0; x < NR; ++x)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    float *o = bs + (x * 32 + 16 * mt + r) * kPitch + 2 * q;
                    *reinterpret_cast<float2 *>(o) = make_float2(acc[x][mt][0], acc[x][mt][1]);
                    *reinterpret_cast<float2 *>(o + 8 * kPitch) = make_float2(acc[x][mt][2], acc[x][mt][3]);
                }
        }
        __syncwarp();
#pragma unroll
        for (int x = 0; x < NR; ++x)
            static_for<N + 1>([&](auto J) { g[x][decltype(J)::value] = bs[(x * 32 + lane) * kPitch + decltype(J)::value]; });
    }
};

// One block tile of the step; every thread of the block calls it. buf, full, empty: the block's
// stage buffers and their mbarriers; nt: tiles this block has stepped before (the buffers'
// phases follow from it: each tile makes kTotal / kStages uses of every buffer). Returns false,
// with LB_HEALTH_TIMEOUT in the health word, when a wait did not end within its bound (warp 0
// then lets the fills it has in flight land before it leaves).
// tm: tensor map of fin (one box per x-row group), or null to copy plane by plane.
// TC (float, one warp per block): the x-row sums of every stage on the tensor cores.
// Ident: the caller's plane order is the library's (no plane table lookups on the stores).
template <class L1, int N, class T, int W, bool FixedX, bool Coherent, bool TC = false, bool Ident = false>
SMRT_D bool tp_block_tile(const TPArgs<T> &a, const TPStepTables<L1, T, false> &s, const T *__restrict__ fin,
                          T *__restrict__ fout, int tile_index, T *buf, unsigned long long *full,
                          unsigned long long *empty, unsigned nt, const CUtensorMap *tm) {
    using C = TPCell<L1, N, T>;
    using S = TPBlockStage<L1, T, W>;
    static_assert(N + 1 <= TPTables<L1, T>::kPow, "the powers table holds e^0 .. e^5");
    static_assert(!TC || (W == 1 && std::is_same<T, float>::value),
                  "tensor-core x-rows: float states, one warp per block (its stage buffer is its scratch)");
    constexpr int Q1 = L1::Q1;
    constexpr int NP1 = L1::NP1;
    constexpr int P2 = Q1 * Q1;
    constexpr int Q = P2 * Q1;
    constexpr int EM = S::kEmax;
    constexpr int SEG = S::kSeg;
    constexpr int NS = S::kStages;
    const int warp = int(threadIdx.x >> 5), lane = int(threadIdx.x & 31);
    const int2 tile = a.tiles[tile_index];
    const InstanceInfo &in = a.inst[tile.x];
    const int x0 = tile.y, x = x0 + 32 * warp + lane, L = in.nx, kx = in.kx;
    const bool active = x < L;
    const long long base = in.cell_off;
    const T *gl = a.ghosts + (long long)tile.x * 2 * Q;
    const T *gr = gl + Q;
    // every plane contributes elements [g_al, g_al + SEG) of itself, clipped to [0, stride)
    const long long g_al = (base + x0 - kx - EM) & ~(long long)(S::kAlign - 1);
    const long long cs = g_al < 0 ? 0 : g_al;
    const long long ce = (g_al + SEG < a.stride) ? g_al + SEG : a.stride;
    const unsigned nbytes = unsigned((ce - cs) * (long long)sizeof(T));
    const int dst_off = int(cs - g_al);
    const unsigned long long u0 = (unsigned long long)nt * (S::kTotal / NS);  // earlier uses of each buffer
    // does any pull of the tile come from beyond the left / right fixed end (block-uniform)?
    const int xmax = (x0 + 32 * W < L ? x0 + 32 * W : L) - 1;
    const bool needL = FixedX && x0 - EM - kx < 0;
    const bool needR = FixedX && xmax + EM - kx >= L;
    // caller plane of library population i
    auto plane = [&](int i) -> long long {
        if constexpr (Ident)
            return i;
        else
            return __ldg(a.plane_idx + i);
    };
    // warp 0: bit b of pending says buffer b has a fill issued and not yet waited for, bit b of
    // fpar is that fill's phase parity
    unsigned pending = 0u, fpar = 0u;
    // warp 0 only: refill the buffer of stage st once every warp has released its previous fill
    auto issue = [&](int st) -> bool {
        const int sb = st % NS;
        const unsigned long long u = u0 + (unsigned long long)(st / NS);  // this fill is use u of buffer sb
        if (u > 0 && !__all_sync(0xffffffffu, mbar_wait(empty + sb, unsigned((u - 1) & 1ull)))) return false;
        pending |= 1u << sb;
        fpar = (fpar & ~(1u << sb)) | (unsigned(u & 1ull) << sb);
        const int cz = st / S::kPerZ, p = st % S::kPerZ;
        const int nplanes = p ? 2 * Q1 : Q1;
        const int k0 = p ? (2 * p - 1) * Q1 : 0;  // in-plane index of the stage's first population
        unsigned long long *b = full + sb;
        T *sbuf = buf + size_t(sb) * S::kStage;
        if constexpr (Coherent) fence_async_global();
        fence_async_shared();
        if (needL || needR) {  // the stage's end-state populations ride along with its fill
            const int i0 = cz * P2 + k0;
            for (int k = lane; k < nplanes; k += 32) {
                T *gs = sbuf + S::kEnds + (k < Q1 ? k : S::kGrp + k - Q1);
                if (needL) cp_async_elem(gs, gl + i0 + k);
                if (needR) cp_async_elem(gs + Q1, gr + i0 + k);
            }
            cp_async_mbar_arrive(b);
            __syncwarp();  // before lane 0's arrival below can complete the phase
        }
        if (tm) {  // one box per row group: d planes (library order) x SEG elements from g_al
            if (lane == 0) {
                mbar_arrive_expect_tx(b, unsigned(nplanes) * unsigned(SEG * sizeof(T)));
                tma_load_2d(sbuf, tm, int(g_al), cz * P2 + k0, b);
                if (p) tma_load_2d(sbuf + S::kGrp, tm, int(g_al), cz * P2 + k0 + Q1, b);
            }
        } else {
            if (lane == 0) mbar_arrive_expect_tx(b, unsigned(nplanes) * nbytes);
            __syncwarp();
            for (int k = lane; k < nplanes; k += 32)  // a pair stage of D1Q17 has 34 planes
                bulk_copy_g2s(sbuf + (k / Q1) * S::kGrp + (k % Q1) * SEG + dst_off,
                              fin + plane(cz * P2 + k0 + k) * a.stride + cs, nbytes, b);
        }
        return true;
    };
    auto fail = [&]() -> bool {
        if (lane == 0) atomicOr(a.health, 2u);
        // warp 0: let the fills still in flight land before the block can leave (each wait bounded)
        for (int q = 0; q < NS; ++q)
            if ((pending >> q) & 1u) mbar_wait(full + q, (fpar >> q) & 1u);
        return false;
    };
    // the lane's pull by x-velocity a of a staged row sits at row + a SEG + tb - e_a; each
    // (plane, slot) is read by this lane only, so the lane may overwrite its own slots
    const int tb = int(base + x - kx - g_al);
    // pulls from beyond the line's ends, by x-velocity (bit a). Fixed ends: such a pull reads the
    // end state staged after the group's rows; a warp none of whose cells has one reads the rows
    // directly. (Rewriting the lanes' slots in the staged rows instead, one diverged branch per
    // velocity and stage, took an edge warp 62 k cycles per tile where the sums take 15 k.) The wrapped
    // pulls of a periodic line, and the operands of the tensor cores, are rewritten in the rows.
    unsigned beyL = 0u, beyR = 0u;
    if (active)
        static_for<Q1>([&](auto A) {
            constexpr int av = decltype(A)::value;
            const int t = x - e1<L1>(av) - kx;
            if (t < 0) beyL |= 1u << av;
            if (t >= L) beyR |= 1u << av;
        });
    const unsigned beyond = beyL | beyR;
    constexpr bool kRewrite = TC || !FixedX;
    const bool edge = !kRewrite && __any_sync(0xffffffffu, beyond != 0u);
    if (warp == 0)
        for (int st = 0; st < NS; ++st)
            if (!issue(st)) return fail();
    TPTensorRows<L1, N> tc;
    if constexpr (TC) {
        static_assert(2 * 32 * TPTensorRows<L1, N>::kPitch <= S::kStage, "scratch fits a stage buffer");
        tc.init(lane, SEG);
    }
    T R[C::M];
    static_for<C::M>([&](auto G) { R[decltype(G)::value] = T(0); });
    T h[N + 1][N + 1];
    static_for<N + 1>([&](auto J) {
        static_for<N + 1 - decltype(J)::value>([&](auto K) { h[decltype(J)::value][decltype(K)::value] = T(0); });
    });
#pragma unroll 1
    for (int st = 0; st < S::kTotal; ++st) {
        const int sb = st % NS;
        const unsigned long long u = u0 + (unsigned long long)(st / NS);
        if (!__all_sync(0xffffffffu, mbar_wait(full + sb, unsigned(u & 1ull)))) return fail();
        pending &= ~(1u << sb);
        const int cz = st / S::kPerZ, p = st % S::kPerZ;
        T *bs = buf + size_t(sb) * S::kStage;
        if (kRewrite && active && beyond) {
            const int nrows = p ? 2 : 1;
            const int k0 = p ? (2 * p - 1) * Q1 : 0;
            static_for<Q1>([&](auto A) {
                constexpr int av = decltype(A)::value;
                if ((beyond >> av) & 1u) {
                    const int t = x - e1<L1>(av) - kx;
                    for (int r = 0; r < nrows; ++r) {
                        T v;
                        if constexpr (FixedX)  // the end state's population, staged with the fill
                            v = bs[r * S::kGrp + S::kEnds + (t < 0 ? 0 : Q1) + av];
                        else
                            v = load_pop<Coherent>(fin + plane(cz * P2 + k0 + r * Q1 + av) * a.stride + base +
                                                   wrap(t, L));
                        bs[r * S::kGrp + av * SEG + tb - e1<L1>(av)] = v;
                    }
                }
            });
            fence_async_shared();  // own slots rewritten: before the buffer's next fill
        }
        if constexpr (TC) {
            __syncwarp();  // the rewritten slots are operands of other lanes
            if (p == 0) {
                float g[1][N + 1];
                tc.template rows<1>(bs, S::kGrp, tb - lane, lane, g);
                if (active) C::yrest(g[0], h);
            } else {
                float g[2][N + 1];
                tc.template rows<2>(bs, S::kGrp, tb - lane, lane, g);
                if (active) C::ypair_pw(g[0], g[1], s.pw[2 * p - 1], h);
            }
            if (active && p == NP1) C::zfold_pw(h, s.pw[cz], R);
            fence_async_shared();  // scratch written and read: before the buffer's next fill
        } else if (active) {
            // at(ic<a>): the stage offset of the lane's pull by x-velocity a in the group of +e_b
            auto sums = [&](auto &&at) {
                if (p == 0) {
                    T g[N + 1];
                    C::xrow([&](auto A) -> T { return bs[at(A)]; }, g);
                    C::yrest(g, h);
                } else {
                    T gp[N + 1], gm[N + 1];
                    if constexpr (std::is_same<T, float>::value) {  // both rows in packed pairs
                        F2 g2[N + 1];
                        TPCell<L1, N, F2>::xrow(
                            [&](auto A) -> F2 {
                                const int o = at(A);
                                return F2(bs[o], bs[o + S::kGrp]);
                            },
                            g2);
                        static_for<N + 1>([&](auto J) {
                            gp[decltype(J)::value] = g2[decltype(J)::value].lo();
                            gm[decltype(J)::value] = g2[decltype(J)::value].hi();
                        });
                    } else {
                        C::xrow([&](auto A) -> T { return bs[at(A)]; }, gp);
                        C::xrow([&](auto A) -> T { return bs[at(A) + S::kGrp]; }, gm);
                    }
                    C::ypair_pw(gp, gm, s.pw[2 * p - 1], h);
                }
            };
            if (edge)
                sums([&](auto A) -> int {
                    constexpr int av = decltype(A)::value;
                    const int inside = tb + av * SEG - e1<L1>(av);
                    const int l = (beyL >> av) & 1u ? S::kEnds + av : inside;
                    return (beyR >> av) & 1u ? S::kEnds + Q1 + av : l;
                });
            else
                sums([&](auto A) -> int { return tb + decltype(A)::value * SEG - e1<L1>(decltype(A)::value); });
            if (p == NP1) C::zfold_pw(h, s.pw[cz], R);
        }
        __syncwarp();  // every lane of this warp is done with buffer sb
        if (lane == 0) mbar_arrive(empty + sb);
        if (warp == 0 && st + NS < S::kTotal && !issue(st + NS)) return fail();
    }
    if (active) {
        if constexpr (!TC) C::x_to_powers(R);  // the tensor-core sums are in powers already
        const bool ok = C::collide_moments(R, T(a.cd), tau_a<T>(in), tau_b<T>(in), in.model, T(in.es_b));
        if (!ok) atomicOr(a.health, 1u);
        C::x_from_powers(R);
        T *dst = fout + base + x;
        auto put = [&](int i, T v) { dst[plane(i) * a.stride] = v; };
#pragma unroll 1
        for (int cz = 0; cz < Q1; ++cz) {
            T Pc[N + 1][N + 1];
            C::template zplane_pw<T>(R, s.pw[cz], Pc);
            const int zc = (cz + 1) >> 1;
            {
                T Pb[N + 1];
                static_for<N + 1>([&](auto J) { Pb[decltype(J)::value] = Pc[decltype(J)::value][0]; });
                C::emit_x(Pb, s.w3[s.row(0, zc)], cz * P2, put);
            }
            // rows (p, zc): a running pointer, or the index, whichever the compiler makes less of (D1Q17-P1 in
            // double, one round of tiles, index against pointer: N = 5 1590 / 1529 us, N = 4 1345 / 1384)
            constexpr bool kIndexed = N < 5;
            const T(*wrow)[NP1 + 1] = s.w3 + s.row(1, zc);
#pragma unroll 1
            for (int p = 1; p <= NP1; ++p) {
                T Pp[N + 1], Pm[N + 1];
                C::template yrows_pw<T>(Pc, s.pw[2 * p - 1], Pp, Pm);
                const T(&w3)[NP1 + 1] = kIndexed ? s.w3[s.row(p, zc)] : *wrow;
                wrow += p < zc ? 1 : p + 1;
                if constexpr (std::is_same<T, float>::value) {  // both rows in packed pairs
                    F2 Pr[N + 1];
                    static_for<N + 1>([&](auto J) { Pr[decltype(J)::value] = F2(Pp[decltype(J)::value], Pm[decltype(J)::value]); });
                    auto put2 = [&](int i, F2 v) {
                        put(i, v.lo());
                        put(i + Q1, v.hi());
                    };
                    TPCell<L1, N, F2>::emit_x(Pr, w3, cz * P2 + (2 * p - 1) * Q1, put2);
                } else {
                    C::emit_x(Pp, w3, cz * P2 + (2 * p - 1) * Q1, put);
                    C::emit_x(Pm, w3, cz * P2 + 2 * p * Q1, put);
                }
            }
        }
    }
    return true;
}

// The block's mbarriers (full[kStages], then empty[kStages]) and stage buffers in dynamic
// shared memory; thread 0 initialises the barriers (published by the block barrier that
// follows in the kernel).
template <class L1, class T, int W>
SMRT_D void tp_block_setup(unsigned char *dyn, unsigned long long *&full, unsigned long long *&empty, T *&buf) {
    using S = TPBlockStage<L1, T, W>;
    full = reinterpret_cast<unsigned long long *>(dyn);
    empty = full + S::kStages;
    buf = reinterpret_cast<T *>(dyn + 128);
    if (threadIdx.x == 0) {
        for (int q = 0; q < S::kStages; ++q) {
            mbar_init(full + q, 1);
            mbar_init(empty + q, W);
        }
        fence_mbar_init();
    }
}

// Blocks of 128 threads per SM that the step kernels leave registers for (0: the compiler's own
// choice). Float: 4 (128 registers) for lines with fixed ends on D1Q9-P1. Without it they take 168
// and three blocks fit: the persistent launch then needs a second, nearly empty round for 572 tiles
// on 152 SMs. Else 3 (168): on D1Q17-P1 three 128-cell blocks fill the shared memory, and the wrapped
// pulls of a periodic line take more registers; 128 of them only made spills there. N = 5 (N = 4), ms
// per step, 128 -> 168: 64 lines of 325 cells on D1Q17-P1 0.316 -> 0.275; 64 periodic lines of 400,
// persistent, D1Q9-P1 0.232 -> 0.144 (0.211 -> 0.140), D1Q17-P1 1.92 -> 1.81 (1.85 -> 1.06).
template <class L1, class T, bool FixedX, bool TC>
constexpr int kTPMinBlocks = std::is_same<T, float>::value && !TC ? (FixedX && L1::Q1 == 9 ? 4 : 3) : 0;

// One step: block b (W warps) takes the block tile b.
// maps: tensor maps of the two states, used when a.tma is set (and the dynamic shared memory
// is 128-byte aligned, as the boxes need).
template <class L1, int N, class T, int W, bool FixedX, bool TC = false, bool Ident = false>
__global__ void __launch_bounds__(128, kTPMinBlocks<L1, T, FixedX, TC>) tp_step_line_block(TPArgs<T> a, int ntiles, const __grid_constant__ TPMaps maps) {
    __shared__ TPStepTables<L1, T, false> s;
    extern __shared__ __align__(128) unsigned char dyn[];
    unsigned long long *full, *empty;
    T *buf;
    tp_block_setup<L1, T, W>(dyn, full, empty, buf);
    tp_load_step_tables<L1>(a, s);  // ends with __syncthreads
    const int t = blockIdx.x;
    if (t >= ntiles) return;
    const CUtensorMap *tm = (a.tma && (smem_addr(dyn) & 127u) == 0u) ? &maps.src : nullptr;
    tp_block_tile<L1, N, T, W, FixedX, false, TC, Ident>(a, s, a.fin, a.fout, t, buf, full, empty, 0u, tm);
}

// All nsteps steps in one cooperative launch (see step_line_persistent in kernels.cuh); the
// blocks stride over the block tiles.
template <class L1, int N, class T, int W, bool FixedX, bool TC = false, bool Ident = false>
__global__ void __launch_bounds__(128, kTPMinBlocks<L1, T, FixedX, TC>) tp_step_line_persistent_block(TPArgs<T> a, int nsteps, int ntiles,
                                                                     unsigned *barg, const __grid_constant__ TPMaps maps) {
    __shared__ TPStepTables<L1, T, false> s;
    __shared__ int failed;
    extern __shared__ __align__(128) unsigned char dyn[];
    unsigned long long *full, *empty;
    T *buf;
    tp_block_setup<L1, T, W>(dyn, full, empty, buf);
    if (threadIdx.x == 0) failed = 0;
    tp_load_step_tables<L1>(a, s);
    unsigned gen = 0;
    if (threadIdx.x == 0) gen = atomicAdd(&barg[1], 0u);
    const unsigned step0 = __ldcg(&barg[2]);
    const T *src = a.fin;
    T *dst = a.fout;
    const bool use_tma = a.tma && (smem_addr(dyn) & 127u) == 0u;
    unsigned nt = 0;  // tiles this block has stepped
    for (int st = 0; st < nsteps; ++st) {
        const CUtensorMap *tm = use_tma ? (src == a.fin ? &maps.src : &maps.dst) : nullptr;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
            if (*static_cast<volatile int *>(&failed)) break;  // another warp gave up
            if (!tp_block_tile<L1, N, T, W, FixedX, true, TC, Ident>(a, s, src, dst, t, buf, full, empty, nt, tm)) {
                failed = 1;
                break;
            }
            ++nt;
        }
        __syncthreads();
        if (failed) return;
        if (st + 1 < nsteps) {
            if (!grid_barrier(barg, gen, a.health)) return;
            const T *nsrc = dst;
            dst = (dst == a.fout) ? const_cast<T *>(a.fin) : a.fout;
            src = nsrc;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) barg[2] = step0 + unsigned(nsteps);
}

// ------------------------------------------------------------------------------ kernels
// ------------------------------------------------------------------ one cell per block
// For problems too small to fill the GPU with one thread per cell (the paper's own runs are
// single shocks of 100 cells), each block takes one cell: its d^3 pulled populations go to
// shared memory, the x-rows and the raw moments are summed by the block's threads, and the
// rebuild is spread over them again. Block b takes cell x0 + b % 32 of the 32-cell tile b / 32.
//
// Float: the moment-space steps run on one thread, whose compile-time constants beat tables.
template <class L1, int N>
struct TPCellShared {
    static constexpr int Q1 = L1::Q1, P2 = Q1 * Q1, Q = P2 * Q1, M = nmom(N);
    float f[Q];             // pulled populations, library order
    float g[P2][N + 1];     // x-row sums g_j of row (b, c) = b + d c
    float ep[Q1][N + 1];    // e_a^j
    float R[M];             // raw moments, then the rebuild coefficients
    float h[Q1][N + 1][N + 1];  // per z-plane c: sum over y of the x-row sums (then of the rebuild)
};

template <class L1, int N, bool FixedX>
__global__ void __launch_bounds__(128) tp_step_cell_kernel(TPArgs<float> a) {
    using C = TPCell<L1, N, float>;
    using SH = TPCellShared<L1, N>;
    constexpr int Q1 = SH::Q1, P2 = SH::P2, Q = SH::Q, M = SH::M;
    __shared__ TPStepTables<L1, float> s;
    __shared__ SH sh;
    tp_load_step_tables<L1>(a, s);  // ends with __syncthreads
    const int tid = threadIdx.x;
    const int2 tile = a.tiles[blockIdx.x >> 5];
    const InstanceInfo &in = a.inst[tile.x];
    const int x = tile.y + int(blockIdx.x & 31u), L = in.nx, kx = in.kx;
    if (x >= L) return;  // the whole block: no barrier follows for it
    const long long base = in.cell_off;
    const float *gl = a.ghosts + (long long)tile.x * 2 * Q;
    const float *gr = gl + Q;
    for (int q = tid; q < Q1 * (N + 1); q += blockDim.x) {
        const int av = q / (N + 1), j = q % (N + 1);
        float p = 1.f;
        for (int r = 0; r < j; ++r) p *= s.e[av];
        sh.ep[av][j] = p;
    }
    // a1: pull every population of the cell
    for (int i = tid; i < Q; i += blockDim.x) {
        const int t = x - e1<L1>(i % Q1) - kx;
        float v;
        if (FixedX && t < 0)
            v = gl[i];
        else if (FixedX && t >= L)
            v = gr[i];
        else
            v = a.fin[(long long)s.plane[i] * a.stride + base + (FixedX ? t : wrap(t, L))];
        sh.f[i] = v;
    }
    __syncthreads();
    // a3, x first: one x-row per thread
    for (int row = tid; row < P2; row += blockDim.x) {
        const float *fr = sh.f + row * Q1;
        float g[N + 1];
        C::xrow([&](auto A) -> float { return fr[decltype(A)::value]; }, g);
        static_for<N + 1>([&](auto J) { sh.g[row][decltype(J)::value] = g[decltype(J)::value]; });
    }
    __syncthreads();
    // ... then y: h_c(j,k) = sum_b g_(b,c)j e_b^k ...
    constexpr int JK = (N + 1) * (N + 1);
    for (int q = tid; q < Q1 * JK; q += blockDim.x) {
        const int c = q / JK, j = (q % JK) / (N + 1), k = q % (N + 1);
        if (j + k > N) continue;
        float acc = 0.f;
        for (int b = 0; b < Q1; ++b) acc = fma(sh.g[b + Q1 * c][j], sh.ep[b][k], acc);
        sh.h[c][j][k] = acc;
    }
    __syncthreads();
    // ... then z: R_(j,k,l) = sum_c h_c(j,k) e_c^l, one moment per thread
    for (int m = tid; m < M; m += blockDim.x) {
        const int j = mi_comp(m, 0), k = mi_comp(m, 1), l = mi_comp(m, 2);
        float acc = 0.f;
        for (int c = 0; c < Q1; ++c) acc = fma(sh.h[c][j][k], sh.ep[c][l], acc);
        sh.R[m] = acc;
    }
    __syncthreads();
    // a2, a4-a6 in warp 0
    if (tid < 32) {
        float R[M];
        static_for<M>([&](auto G) { R[decltype(G)::value] = sh.R[decltype(G)::value]; });
        C::x_to_powers(R);
        const bool ok = C::collide_moments(R, float(a.cd), tau_a<float>(in), tau_b<float>(in), in.model, float(in.es_b));
        C::x_from_powers(R);
        __syncwarp();
        if (tid == 0) {
            if (!ok) atomicOr(a.health, 1u);
            static_for<M>([&](auto G) { sh.R[decltype(G)::value] = R[decltype(G)::value]; });
        }
    }
    __syncthreads();
    // a7 + a8: z first, Pc_c(j,k) = sum_l P_(j,k,l) e_c^l ...
    for (int q = tid; q < Q1 * JK; q += blockDim.x) {
        const int c = q / JK, j = (q % JK) / (N + 1), k = q % (N + 1);
        if (j + k > N) continue;
        float acc = 0.f;
        for (int l = 0; l + j + k <= N; ++l) acc = fma(sh.R[mi_pos(j, k, l)], sh.ep[c][l], acc);
        sh.h[c][j][k] = acc;
    }
    __syncthreads();
    // ... then one x-row per thread, Pb_j = sum_k Pc_c(j,k) e_b^k, stored as it is formed
    float *dst = a.fout + base + x;
    auto put = [&](int i, float v) { dst[(long long)s.plane[i] * a.stride] = v; };
    for (int row = tid; row < P2; row += blockDim.x) {
        const int b = row % Q1, c = row / Q1;
        float Pb[N + 1];
        static_for<N + 1>([&](auto J) {
            constexpr int j = decltype(J)::value;
            float acc = 0.f;
            static_for<N + 1 - j>([&](auto K) {
                constexpr int k = decltype(K)::value;
                acc = fma(sh.h[c][j][k], sh.ep[b][k], acc);
            });
            Pb[j] = acc;
        });
        C::emit_x(Pb, s.w3[s.row((b + 1) >> 1, (c + 1) >> 1)], row * Q1, put);
    }
}

// Double: every stage is spread over the block's threads, the moment-space steps as the sparse
// stages of lane_cell.cuh on two warps (a full-warp FP64 instruction holds a quarter of the SM's
// FP64 pipe for 64 cycles whether or not its lanes do useful work, so what counts is the number of
// instructions in a row, not the number of lanes they use). One 100-cell shock, N = 5: 46 us per
// step with the moment space on one warp in dense order blocks, 22.8 us here (371 us on the
// block-staged kernel); 4800 cells 204 us (373).
struct TPCellGroup {
    static constexpr int G = 64;
    int lane;
    SMRT_D void sync() const { asm volatile("bar.sync 1, 64;" ::: "memory"); }
};
template <class L1, int N>
struct TPLaneShared {
    static constexpr int Q1 = L1::Q1, P2 = Q1 * Q1, Q = P2 * Q1, M = nmom(N);
    static constexpr int kJK = (N + 1) * (N + 2) / 2;  // (j, k) with j + k <= N
    using C = LaneCell<N>;
    LaneMoments<N> m;
    double f[(Q + 1) / 2 * 2];      // populations, library order
    double g[P2][N + 1];            // x-row sums g_j of row b + d c; x-row coefficients of the rebuild
    double pw[Q1][N + 1];           // e_a^j
    double w[Q1 + 1];
    double h[Q1][kJK];              // per z-plane c: sums over y; plane coefficients of the rebuild
    double cp[N + 1 + (N & 1 ? 0 : 1)];
    double V[C::kForward];
    // (j, k) of index r, j ascending then k, three bits each
    SMRT_HD static constexpr unsigned long long packed(bool second) {
        unsigned long long v = 0;
        int r = 0;
        for (int j = 0; j <= N; ++j)
            for (int k = 0; k + j <= N; ++k, ++r) v |= (unsigned long long)(second ? k : j) << (3 * r);
        return v;
    }
    SMRT_D static int j_of(int r) {
        constexpr unsigned long long v = packed(false);
        return int((v >> (3 * r)) & 7ull);
    }
    SMRT_D static int k_of(int r) {
        constexpr unsigned long long v = packed(true);
        return int((v >> (3 * r)) & 7ull);
    }
    SMRT_D static int jk(int j, int k) { return j * (N + 1) - j * (j - 1) / 2 + k; }
    // The sums of the populations in f: c-scaled raw moments into R (shared). All threads of the
    // block; ends with a block barrier.
    SMRT_D void project(double *R) {
        using T = TPCell<L1, N, double>;
        for (int row = threadIdx.x; row < P2; row += blockDim.x) {
            const double *fr = f + row * Q1;
            double gr[N + 1];
            T::xrow([&](auto A) -> double { return fr[decltype(A)::value]; }, gr);
            if constexpr (N >= 5) gr[5] = fma(120.0, gr[5], fma(30.0, gr[3], gr[1]));  // to powers of e
            gr[4] = fma(12.0, gr[4], gr[2]);
            gr[3] = fma(6.0, gr[3], gr[1]);
            static_for<N + 1>([&](auto J) { g[row][decltype(J)::value] = gr[decltype(J)::value]; });
        }
        __syncthreads();
        // y, +-e_b folded: h_c(j,k) = sum_b g_(b,c)j e_b^k
        for (int q = threadIdx.x; q < Q1 * kJK; q += blockDim.x) {
            const int c = q / kJK, r = q % kJK, j = j_of(r), k = k_of(r);
            double acc = k == 0 ? g[Q1 * c][j] : 0.0;
#pragma unroll
            for (int p = 0; p < L1::NP1; ++p) {
                const double gp = g[Q1 * c + 2 * p + 1][j], gm = g[Q1 * c + 2 * p + 2][j];
                acc = fma(pw[2 * p + 1][k], (k & 1) ? gp - gm : gp + gm, acc);
            }
            h[c][r] = acc;
        }
        __syncthreads();
        // z, +-e_c folded: one moment per thread
        for (int q = threadIdx.x; q < M; q += blockDim.x) {
            const int r = jk(m.comp[q][0], m.comp[q][1]), l = m.comp[q][2];
            double acc = l == 0 ? h[0][r] : 0.0;
#pragma unroll
            for (int p = 0; p < L1::NP1; ++p) {
                const double hp = h[2 * p + 1][r], hm = h[2 * p + 2][r];
                acc = fma(pw[2 * p + 1][l], (l & 1) ? hp - hm : hp + hm, acc);
            }
            R[q] = acc * cp[m.ord[q]];
        }
        __syncthreads();
    }
    // Populations from the (c-scaled) coefficients P (shared): put(i, value without the weights).
    // All threads; P ready on entry.
    template <class Put>
    SMRT_D void rebuild(const double *P, Put &&put) {
        for (int q = threadIdx.x; q < Q1 * kJK; q += blockDim.x) {
            const int c = q / kJK, r = q % kJK, j = j_of(r), k = k_of(r);
            double acc = P[mi_pos(j, k, 0)];
            for (int l = 1; l + j + k <= N; ++l) acc = fma(P[mi_pos(j, k, l)], pw[c][l], acc);
            h[c][r] = acc;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < P2 * (N + 1); q += blockDim.x) {
            const int row = q % P2, j = q / P2, b = row % Q1, c = row / Q1, r = jk(j, 0);
            double acc = h[c][r];
            for (int k = 1; k + j <= N; ++k) acc = fma(h[c][r + k], pw[b][k], acc);
            g[row][j] = acc;
        }
        __syncthreads();
        // one +-e_a pair (or the rest velocity) of a row per thread
        for (int q = threadIdx.x; q < P2 * (L1::NP1 + 1); q += blockDim.x) {
            const int row = q % P2, p = q / P2;
            const double *G = g[row];
            if (p == L1::NP1) {
                put(row * Q1, G[0]);
            } else {
                const double *e = pw[2 * p + 1];
                double ev = fma(e[2], G[2], G[0]), od = e[1] * G[1];
                od = fma(e[3], G[3], od);
                ev = fma(e[4], G[4], ev);
                if constexpr (N >= 5) od = fma(e[5], G[5], od);
                put(row * Q1 + 2 * p + 1, ev + od);
                put(row * Q1 + 2 * p + 2, ev - od);
            }
        }
    }
    // tables of the block (no barrier)
    SMRT_D void load(const TPArgs<double> &a) {
        lane_copy(m, lane_moments<N>());
        if (threadIdx.x < Q1) {
            const double ea = e1<L1>(threadIdx.x);
            double p = 1.0;
            for (int k = 0; k <= N; ++k, p *= ea) pw[threadIdx.x][k] = p;
            w[threadIdx.x] = a.w1[threadIdx.x];
        } else if (threadIdx.x == 32) {
            double p = 1.0;
            for (int k = 0; k <= N; ++k, p *= a.cd) cp[k] = p;
        }
    }
    // the cell's pulled populations and the tables, all in flight together (no barrier)
    template <bool FixedX, class Plane>
    SMRT_D void pull(const TPArgs<double> &a, const double *gl, int x, int L, int kx, Plane &&plane) {
        constexpr int kPer = (Q + 127) / 128;
        double v[kPer];
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
            const int i = threadIdx.x + 128 * r;
            v[r] = 0.0;
            if (i < Q) {
                const int t = x - e1<L1>(i % Q1) - kx;
                if (FixedX && t < 0)
                    v[r] = gl[i];
                else if (FixedX && t >= L)
                    v[r] = gl[Q + i];
                else
                    v[r] = a.fin[plane(i) + (FixedX ? t : wrap(t, L))];
            }
        }
        load(a);
#pragma unroll
        for (int r = 0; r < kPer; ++r)
            if (threadIdx.x + 128 * r < Q) f[threadIdx.x + 128 * r] = v[r];
    }
    SMRT_D double weight(int i) const { return w[i % Q1] * w[i / Q1 % Q1] * w[i / P2]; }
};

template <class L1, int N, bool FixedX>
__global__ void __launch_bounds__(128) tp_step_cell_lanes(TPArgs<double> a) {
    using SH = TPLaneShared<L1, N>;
    constexpr int Q1 = SH::Q1, Q = SH::Q;
    __shared__ __align__(16) unsigned char raw[sizeof(SH)];
    SH &s = *reinterpret_cast<SH *>(raw);
    const int tid = threadIdx.x;
    const int2 tile = a.tiles[blockIdx.x >> 5];
    const InstanceInfo &in = a.inst[tile.x];
    const int x = tile.y + int(blockIdx.x & 31u), L = in.nx, kx = in.kx;
    if (x >= L) return;  // the whole block
    const long long base = in.cell_off;
    const double *gl = a.ghosts + (long long)tile.x * 2 * Q;
    auto plane = [&](int i) -> long long { return (a.ident ? i : __ldg(a.plane_idx + i)) * a.stride + base; };
    s.template pull<FixedX>(a, gl, x, L, kx, plane);
    __syncthreads();
    s.project(s.V + LaneCell<N>::oRc);
    double *P = s.V + LaneCell<N>::oTa;
    if (tid < TPCellGroup::G) {
        const TPCellGroup g{tid};
        LaneCell<N> cell;
        const bool ok = cell.collide(s.m, g, s.V, in.tauA, in.tauB, in.model, in.es_b,
                                     [&](int k, double c) { P[k] = c * s.cp[s.m.ord[k]]; });
        if (tid == 0 && !ok) atomicOr(a.health, 1u);
    }
    __syncthreads();
    double *dst = a.fout + x;
    s.rebuild(P, [&](int i, double c) { dst[plane(i)] = c * s.weight(i); });
}

// lb_moments on the same blocks (double; the small problems above). The paper's 100-cell shock:
// 208 -> 20 us, one thread per cell being 4 warps on the whole GPU.
template <class L1, int N, bool FixedX>
__global__ void __launch_bounds__(128) tp_moments_cell_lanes(TPArgs<double> a, double *out, long long ncells, unsigned mask) {
    using SH = TPLaneShared<L1, N>;
    using C = LaneCell<N>;
    __shared__ __align__(16) unsigned char raw[sizeof(SH)];
    SH &s = *reinterpret_cast<SH *>(raw);
    const int2 tile = a.tiles[blockIdx.x >> 5];
    const InstanceInfo &in = a.inst[tile.x];
    const int x = tile.y + int(blockIdx.x & 31u), L = in.nx, kx = in.kx;
    if (x >= L) return;  // the whole block
    const long long base = in.cell_off;
    s.template pull<FixedX>(a, a.ghosts + (long long)tile.x * 2 * SH::Q, x, L, kx, [&](int i) -> long long {
        return (a.ident ? i : __ldg(a.plane_idx + i)) * a.stride + base;
    });
    __syncthreads();
    s.project(s.V + C::oRc);
    if (threadIdx.x >= TPCellGroup::G) return;
    const TPCellGroup g{int(threadIdx.x)};
    C cell;
    cell.local(s.m, g, s.V);
    if (threadIdx.x != 0) return;
    const double up[3] = {cell.u[0] + a.cd * in.kx, cell.u[1], cell.u[2]};
    double v[C::M];
    for (int p = 0; p < C::M; ++p) v[p] = s.V[C::oTd + p];
    store_moments<N, double>(out, ncells, base + x, mask, cell.rho, up, cell.th, v);
}

// lb_moments of the pulled (pre-collision) populations.
template <class L1, int N, class T>
__global__ void __launch_bounds__(128) tp_moments_kernel(TPArgs<T> a, double *out, long long ncells,
                                                         unsigned mask, int fixedx) {
    __shared__ TPTables<L1, T> s;
    tp_load_tables<L1>(a, s);
    using C = TPCell<L1, N, T>;
    constexpr int Q1 = L1::Q1;
    constexpr int Q = Q1 * Q1 * Q1;
    const int2 tile = a.tiles[blockIdx.x];
    const InstanceInfo &in = a.inst[tile.x];
    const int x = tile.y + threadIdx.x;
    const int L = in.nx;
    if (x >= L) return;
    const long long base = in.cell_off;
    const T *gl = a.ghosts + (long long)tile.x * 2 * Q;
    const T *gr = gl + Q;
    int xs[Q1];
    static_for<Q1>([&](auto A) {
        constexpr int av = decltype(A)::value;
        xs[av] = x - (e1<L1>(av) + in.kx);
    });
    auto pop = [&](int i, auto A) -> T {
        const int t = xs[decltype(A)::value];
        if (fixedx && t < 0) return gl[i];
        if (fixedx && t >= L) return gr[i];
        return a.fin[(long long)s.plane[i] * a.stride + base + wrap(t, L)];
    };
    T R[C::M];
    C::project(pop, s.e, R);
    const T c = T(a.cd);
    T cp[N + 1];
    cp[0] = T(1);
    static_for<N>([&](auto J) { cp[decltype(J)::value + 1] = cp[decltype(J)::value] * c; });
    static_for<C::M>([&](auto G) { R[decltype(G)::value] *= cp[mi_order(decltype(G)::value)]; });
    const T rhom1 = R[0], rho = T(1) + rhom1, ir = rcp(rho);
    const T u[3] = {R[mi_pos(1, 0, 0)] * ir, R[mi_pos(0, 1, 0)] * ir, R[mi_pos(0, 0, 1)] * ir};
    const T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const T thm1 = (R[mi_pos(2, 0, 0)] + R[mi_pos(0, 2, 0)] + R[mi_pos(0, 0, 2)] - T(3) * rhom1 - rho * uu) *
                   ir * T(1.0 / 3.0);
    const T theta = T(1) + thm1;
    T v[C::M];
    static_for<C::M>([&](auto A) {
        constexpr int al = decltype(A)::value;
        T acc = T(0);
        static_for<C::M>([&](auto G) {
            constexpr int g = decltype(G)::value;
            constexpr double h = hdiv(al, g);
            if constexpr (h != 0.0) acc = fma(T(h), R[g], acc);
        });
        v[al] = acc;
    });
    v[0] = rho;
    to_local_divided<N, T>(v, u, theta, thm1);
    const double up[3] = {double(u[0]) + a.cd * in.kx, double(u[1]), double(u[2])};
    store_moments<N, T>(out, ncells, base + x, mask, double(rho), up, double(theta), v);
}

// Equilibrium fill: df = order-N equilibrium of (rho, u_phys - u_bar, theta) minus w_i,
// formed in double and stored as T.
template <class L1, int N, class T>
__global__ void __launch_bounds__(128) tp_fill_kernel(TPArgs<T> a, const double *rho, const double *u,
                                                      const double *theta, long long ncells) {
    __shared__ TPTables<L1, double> s;
    tp_load_tables<L1>(a, s);
    using C = TPCell<L1, N, double>;
    const int2 tile = a.tiles[blockIdx.x];
    const InstanceInfo &in = a.inst[tile.x];
    const int x = tile.y + threadIdx.x;
    if (x >= in.nx) return;
    const long long cell = in.cell_off + x;
    const double uu[3] = {u[cell] - a.cd * in.kx, u[ncells + cell], u[2 * ncells + cell]};
    double P[C::M];
    C::template equilibrium<double>(rho[cell], uu, theta[cell], a.cd, P);
    T *dst = a.fout + cell;
    C::template rebuild<double>(P, s.e, s.w, [&](int i, double v) { dst[(long long)s.plane[i] * a.stride] = T(v); });
}

// End-state populations of every instance, library order: thread t = 2 j + side.
template <class L1, int N, class T>
__global__ void __launch_bounds__(64) tp_ghost_kernel(TPArgs<T> a, const double *states, int ninst, T *ghosts) {
    __shared__ TPTables<L1, double> s;
    tp_load_tables<L1>(a, s);
    using C = TPCell<L1, N, double>;
    constexpr int Q = L1::Q1 * L1::Q1 * L1::Q1;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2 * ninst) return;
    const int j = t / 2;
    const double *st = states + 5 * t;
    const double uu[3] = {st[1] - a.cd * a.inst[j].kx, st[2], st[3]};
    double P[C::M];
    C::template equilibrium<double>(st[0], uu, st[4], a.cd, P);
    T *g = ghosts + (long long)t * Q;
    C::template rebuild<double>(P, s.e, s.w, [&](int i, double v) { g[i] = T(v); });
}

}  // namespace smrt
