// lane_tables.cuh -- compile-time tables for running one cell's SMRT step or its adjoint
// (Yan & Shan, arXiv 2401.11086) on a group of lanes (lane_cell.cuh).
//
// Every linear stage of the cell (sums over the sign orbits, Hermite conversions, binomial passes,
// traces and delta products) is a small sparse matrix with constant structure. It is tabulated here
// as rows of (column, coefficient); a group of lanes takes one row each. Rows are ordered by
// descending length, so that the lanes of one round do about the same number of terms.
#pragma once

#include "lattices.cuh"
#include "moment_tables.cuh"

namespace smrt {

// Sparse rows: row r (r < kRows) writes slot at[r].id from the terms [beg, beg + len).
struct alignas(4) RowAt {  // one 4-byte load
    unsigned short beg = 0;
    unsigned char len = 0, id = 0;
};
template <int ROWS, int NNZ>
struct SparseRows {
    static constexpr int kRows = ROWS, kNnz = NNZ;
    double val[NNZ > 0 ? NNZ : 1] = {};
    RowAt at[ROWS] = {};
    unsigned char col[NNZ > 0 ? NNZ : 1] = {};
    unsigned char row[ROWS] = {};  // the row of a slot
};
// ... whose coefficient is entry j[] of a small run-time vector (the Maxwellian factors G)
template <int ROWS, int NNZ>
struct SparsePass {
    static constexpr int kRows = ROWS, kNnz = NNZ;
    RowAt at[ROWS] = {};
    unsigned char col[NNZ] = {}, j[NNZ] = {};
};

// Fill rows in descending length from a dense predicate. coef(row, col) -> value (0: no term).
template <class Tab, class F>
constexpr void fill_rows(Tab &t, int cols, F coef) {
    int n[Tab::kRows] = {};
    int most = 0;
    for (int r = 0; r < Tab::kRows; ++r) {
        for (int c = 0; c < cols; ++c) n[r] += coef(r, c) != 0.0;
        most = n[r] > most ? n[r] : most;
    }
    int out = 0, at = 0;
    for (int len = most; len >= 0; --len)
        for (int r = 0; r < Tab::kRows; ++r) {
            if (n[r] != len) continue;
            t.at[out].id = (unsigned char)r;
            t.row[r] = (unsigned char)out;
            t.at[out].len = (unsigned char)len;
            t.at[out].beg = (unsigned short)at;
            for (int c = 0; c < cols; ++c) {
                const double v = coef(r, c);
                if (v == 0.0) continue;
                t.col[at] = (unsigned char)c;
                t.val[at++] = v;
            }
            ++out;
        }
}
template <class Tab, class F>
constexpr void fill_pass(Tab &t, int cols, F power) {  // power(row, col) -> j > 0, or 0: no term
    int n[Tab::kRows] = {};
    int most = 0;
    for (int r = 0; r < Tab::kRows; ++r) {
        for (int c = 0; c < cols; ++c) n[r] += power(r, c) != 0;
        most = n[r] > most ? n[r] : most;
    }
    int out = 0, at = 0;
    for (int len = most; len >= 0; --len)
        for (int r = 0; r < Tab::kRows; ++r) {
            if (n[r] != len) continue;
            t.at[out].id = (unsigned char)r;
            t.at[out].len = (unsigned char)len;
            t.at[out].beg = (unsigned short)at;
            for (int c = 0; c < cols; ++c) {
                const int j = power(r, c);
                if (j == 0) continue;
                t.col[at] = (unsigned char)c;
                t.j[at++] = (unsigned char)j;
            }
            ++out;
        }
}

// ------------------------------------------------------------------ moment space
// Sizes of the sparse stages: Hermite conversions (nonzero hfull entries), binomial passes
// (sum of one component over all slots), traces (three terms per slot of order <= N - 2).
template <int N>
constexpr int hermite_nnz() {  // per component: x^j in He_n for j <= n of its parity
    const SlotIndex<N> s;
    int n = 0;
    for (int a = 0; a < nmom(N); ++a) {
        int m = 1;
        for (int k = 0; k < 3; ++k) m *= s.c[a][k] / 2 + 1;
        n += m;
    }
    return n;
}
template <int N>
constexpr int pass_nnz() {
    const SlotIndex<N> s;
    int n = 0;
    for (int a = 0; a < nmom(N); ++a) n += s.c[a][0];
    return n;
}

template <int N>
struct alignas(16) LaneMoments {
    static constexpr int M = nmom(N);
    static constexpr int M2 = nmom(N - 2);            // slots of order <= N - 2
    static constexpr int M4 = N >= 4 ? nmom(N - 4) : 1;  // slots of order <= N - 4
    static constexpr int kH = hermite_nnz<N>(), kP = pass_nnz<N>();
    static constexpr int kC = (N - 1) * (N / 2 + 1);  // C[n][j] in a (N / 2 + 1)-wide table
    SparseRows<M, kH> hd, hf, hdT, hfT;  // sum_g hdiv(a,g) x_g, sum_g hfull(a,g) x_g, and transposes
    SparsePass<M, kP> pass[3], passT[3];
    SparseRows<M2, 3 * M2> tr;           // (tr X)_p of the order p + 2, p of order <= N - 2
    SparseRows<M, 3 * M2> trT;           // its transpose
    SparseRows<M, 3 * M2> del;           // (delta Y)_p, p of order 2..N, Y of order p - 2
    SparseRows<M2, 3 * M2> delT;         // its transpose
    SparseRows<kC, kC * (N / 2 + 1)> cj; // C[n][j] = sum_m B(n,m) D(n-2m, j-m) s_(n,m)
    SparseRows<ntau(N), kC * (N / 2 + 1)> cjT;
    unsigned char ord[M] = {}, comp[M][4] = {};  // order, components of a slot
    // ES-BGK target of order 4: ordered pairs of order-2 slots adding up to the slot
    unsigned char es_n[M] = {}, es_q1[M][8] = {}, es_q2[M][8] = {};
    // pairs of slots p = q + j e_k, by j: pairs [gbeg[j], gbeg[j + 1]) of gp[k], gq[k]
    unsigned char gp[3][kP] = {}, gq[3][kP] = {};
    unsigned short gbeg[N + 2] = {};
    SMRT_HD static constexpr int c_slot(int n, int j) { return (n - 2) * (N / 2 + 1) + j; }
    constexpr LaneMoments() {
        const SlotIndex<N> s;
        for (int p = 0; p < M; ++p) {
            ord[p] = (unsigned char)s.ord[p];
            for (int k = 0; k < 3; ++k) comp[p][k] = (unsigned char)s.c[p][k];
        }
        double h1[N + 1][N + 1] = {}, fa[N + 1] = {};
        for (int n = 0; n <= N; ++n) {
            fa[n] = fact_small(n);
            for (int j = 0; j <= n; ++j) h1[n][j] = he_coef_l(n, j);
        }
        auto he = [&](int a, int g) {  // hfull
            return h1[s.c[a][0]][s.c[g][0]] * h1[s.c[a][1]][s.c[g][1]] * h1[s.c[a][2]][s.c[g][2]];
        };
        auto af = [&](int a) { return fa[s.c[a][0]] * fa[s.c[a][1]] * fa[s.c[a][2]]; };
        fill_rows(hd, M, [&](int a, int g) { return he(a, g) / af(a); });
        fill_rows(hf, M, [&](int a, int g) { return he(a, g); });
        fill_rows(hdT, M, [&](int g, int a) { return he(a, g) / af(a); });
        fill_rows(hfT, M, [&](int g, int a) { return he(a, g); });
        for (int k = 0; k < 3; ++k) {
            auto up = [&](int p, int q) {  // p = q + j e_k, j > 0
                for (int d = 0; d < 3; ++d)
                    if (d != k && s.c[p][d] != s.c[q][d]) return 0;
                return s.c[p][k] > s.c[q][k] ? s.c[p][k] - s.c[q][k] : 0;
            };
            fill_pass(pass[k], M, up);
            fill_pass(passT[k], M, [&](int q, int p) { return up(p, q); });
            int at = 0;
            for (int j = 1; j <= N; ++j) {
                gbeg[j] = (unsigned short)at;
                for (int p = 0; p < M; ++p)
                    for (int q = 0; q < M; ++q)
                        if (up(p, q) == j) {
                            gp[k][at] = (unsigned char)p;
                            gq[k][at++] = (unsigned char)q;
                        }
            }
            gbeg[N + 1] = (unsigned short)at;
        }
        auto plus2 = [&](int q, int p) {  // the axis k with q = p + 2 e_k, or -1
            for (int k = 0; k < 3; ++k) {
                bool same = s.c[q][k] == s.c[p][k] + 2;
                for (int d = 0; d < 3; ++d) same = same && (d == k || s.c[q][d] == s.c[p][d]);
                if (same) return k;
            }
            return -1;
        };
        auto trc = [&](int p, int q) {
            const int k = plus2(q, p);
            return k < 0 ? 0.0 : double((s.c[p][k] + 2) * (s.c[p][k] + 1));
        };
        auto dlc = [&](int q, int p) {
            const int r = s.ord[q];
            return plus2(q, p) < 0 ? 0.0 : 1.0 / double(r * (r - 1));
        };
        fill_rows(tr, M, trc);
        fill_rows(trT, M2, [&](int q, int p) { return trc(p, q); });
        fill_rows(del, M2, dlc);
        fill_rows(delT, M, [&](int p, int q) { return dlc(q, p); });
        auto bd = [&](int c, int t) {  // coefficient of s_t in C slot c
            const int n = c / (N / 2 + 1) + 2, j = c % (N / 2 + 1);
            if (j > n / 2) return 0.0;
            for (int m = 0; m <= j; ++m)
                if (tau_slot(n, m) == t) return coefB(n, m) * coefD(n - 2 * m, j - m);
            return 0.0;
        };
        fill_rows(cj, ntau(N), bd);
        fill_rows(cjT, kC, [&](int t, int c) { return bd(c, t); });
        const EsTables<N> es;
        for (int p = 0; p < M; ++p) {
            es_n[p] = (unsigned char)es.n[p];
            for (int i = 0; i < 8; ++i) {
                es_q1[p][i] = (unsigned char)es.q1[p][i];
                es_q2[p][i] = (unsigned char)es.q2[p][i];
            }
        }
    }
};

// ------------------------------------------------------------------ sums over the populations
// A cell's populations x_i are first transformed in place: x[2p+1], x[2p+2] become the sum and the
// difference of pair p, then the sums (and the differences) of an orbit's pairs their
// Walsh-Hadamard transform, entry c of which sits at the pair of the orbit's member c.
template <class Lat, int N>
constexpr int orbit_nnz() {
    const SignOrbits<Lat> s;
    int n = 1;
    for (int o = 0; o < s.n; ++o)
        for (int g = 0; g < nmom(N); ++g) n += s.monomial(o, g) != 0;
    return n;
}
template <class Lat, int N>
struct alignas(16) LaneOrbits {
    static constexpr int M = nmom(N), Q = Lat::Q, NP = Lat::NP;
    static constexpr int kNnz = orbit_nnz<Lat, N>();
    SparseRows<M, kNnz> raw;   // R_g from the transformed populations
    SparseRows<Q, kNnz> rawT;  // the transposed sums, in transformed form
    signed char ex[Q] = {};                // x component of population i
    unsigned char flip[NP] = {};           // the pair's member is -e of the pair
    int n0 = 0, n1 = 0;                    // butterflies (pair, pair) of the two transform steps
    unsigned char b0[NP][2] = {}, b1[NP][2] = {};
    constexpr LaneOrbits() {
        const SignOrbits<Lat> s;
        for (int o = 0; o < s.n; ++o) {
            const int np = 1 << (s.k[o] - 1);
            for (int b = 0; b < np; ++b) flip[s.pair[o][b]] = (unsigned char)s.flip[o][b];
            for (int b = 0; b < np; ++b) {
                if (np >= 2 && !(b & 1)) {
                    b0[n0][0] = (unsigned char)s.pair[o][b];
                    b0[n0++][1] = (unsigned char)s.pair[o][b | 1];
                }
                if (np >= 4 && !(b & 2)) {
                    b1[n1][0] = (unsigned char)s.pair[o][b];
                    b1[n1++][1] = (unsigned char)s.pair[o][b | 2];
                }
            }
        }
        for (int p = 0; p < NP; ++p) {
            ex[2 * p + 1] = (signed char)Lat::e(p, 0);
            ex[2 * p + 2] = (signed char)-Lat::e(p, 0);
        }
        int owner[NP] = {}, bit[NP] = {};
        for (int o = 0; o < s.n; ++o)
            for (int b = 0; b < (1 << (s.k[o] - 1)); ++b) owner[s.pair[o][b]] = o, bit[s.pair[o][b]] = b;
        int mono[NP][M] = {}, cls[NP][M] = {}, odd[M] = {};
        for (int o = 0; o < s.n; ++o)
            for (int g = 0; g < M; ++g) mono[o][g] = s.monomial(o, g), cls[o][g] = s.parity_class(o, g);
        for (int g = 0; g < M; ++g) odd[g] = mi_order(g) & 1;
        auto co = [&](int g, int i) {
            if (i == 0) return g == 0 ? 1.0 : 0.0;
            const int p = (i - 1) / 2, o = owner[p];
            return (odd[g] == ((i - 1) & 1) && cls[o][g] == bit[p]) ? double(mono[o][g]) : 0.0;
        };
        fill_rows(raw, Q, co);
        fill_rows(rawT, M, [&](int i, int g) { return co(g, i); });
    }
};

}  // namespace smrt
