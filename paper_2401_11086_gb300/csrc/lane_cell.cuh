// lane_cell.cuh -- one cell's SMRT collision and its adjoint on a group of lanes, in double.
//
// Why. A double-precision instruction occupies an SM sub-partition of this GPU for 64 cycles (76
// when all four of an SM run) whether 1 or 32 lanes of the warp need it, and a thread's next one
// waits for it. A thread that owns a cell therefore takes (instructions per cell) x 64 cycles
// however small the grid is: 669 instructions, 21 us, per step of a D3Q39 shock; 4.7 k, 150 us,
// per adjoint step on D3Q103. On a small grid most of the GPU idles meanwhile. Here the cell's
// moments and populations sit in shared memory and the lanes of a group share every stage, so the
// work of the grid spreads over all sub-partitions with full warps.
//
// The stages are those of core.cuh and adjoint.cuh (the same formulas in the divided form), each a
// sparse matrix of lane_tables.cuh. Group supplies lane, G (lanes of the group) and sync().
// Vectors are addressed by their offset in the cell's array V.
#pragma once

#include "lane_tables.cuh"

namespace smrt {

template <int N>
struct LaneCell {
    static constexpr int M = nmom(N), M2 = LaneMoments<N>::M2, M4 = LaneMoments<N>::M4;
    static constexpr int KT = ntau(N), KC = LaneMoments<N>::kC;
    using Tab = LaneMoments<N>;
    double rho, rhom1, ir, u[3], uu, thm1, th;  // scalars every lane holds

    // vectors of a cell in V (doubles)
    enum : int {
        oRc = 0,                                 // raw moments, c^|g| R_g
        oPw = oRc + M,                           // theta^(-j/2), then theta^(j/2), j <= N
        oG = oPw + 2 * (N + 1),                  // G[sign][axis][j]
        oS = oG + 6 * (N + 1),                   // s_k, then R_k = 1 / (A_k + B_k rho)
        oC = oS + 2 * KT,                        // C[n][j]
        oTa = oC + KC, oP1 = oTa + M, oP2 = oP1 + M, oTd = oP2 + M,
        oT1 = oTd + M, oT2 = oT1 + M2, oZ = oT2 + M4,
        oTdp = oZ + M2, oY = oTdp + M, oQ1 = oY + M, oQ2 = oQ1 + M,
        kForward = (oQ2 + M + 1) / 2 * 2,
        // adjoint
        oLc = kForward, oTapb = oLc + M, oQ2b = oTapb + M, oQ1b = oQ2b + M, oYb = oQ1b + M,
        oTdpb = oYb + M, oW1 = oTdpb + M, oW2 = oW1 + M2, oX1 = oW2 + M4, oTdb = oX1 + M2,
        oP3b = oTdb + M, oP2b = oP3b + M, oP1b = oP2b + M, oTab = oP1b + M,
        oA = oTab + M, oE = oA + N + 1,          // sums per order: tdpb.tdp, tdb.td
        oGb = oE + N + 1,                        // G's adjoints [sign][axis][j]
        oMx = oGb + 6 * (N + 1),                 // per (sign, axis): adjoints of u and theta
        oCb = oMx + 12, oSr = oCb + KC,          // C's adjoints; the s_k's part of rho's adjoint
        oTau = oSr + KT,                         // relaxation-time gradients
        kAdjoint = (oTau + KT + 1) / 2 * 2
    };

    // acc + sum of the products term(i) gives, i < n. The next term is loaded before the current
    // product is issued, so that the loads' latency runs under the multiply-add.
    template <class Term>
    SMRT_HD static double dot(int n, double acc, Term &&term) {
        double v = 0.0, y = 0.0;
        if (n > 0) term(0, v, y);
        for (int i = 0; i < n; ++i) {
            const double cv = v, cy = y;
            if (i + 1 < n) term(i + 1, v, y);
            acc = fma(cv, cy, acc);
        }
        return acc;
    }
    template <class Rows>
    SMRT_HD static double row_dot(const Rows &t, const RowAt &r, const double *x) {
        const int b = r.beg;
        return dot(r.len, 0.0, [&](int i, double &v, double &y) {
            y = x[t.col[b + i]];
            v = t.val[b + i];
        });
    }
    template <class Rows, class Group, class Put>
    SMRT_HD static void rows(const Rows &t, const Group &g, const double *x, Put &&put, int below = 1 << 30) {
        for (int r = g.lane; r < Rows::kRows; r += Group::G) {
            const RowAt at = t.at[r];
            if (at.id < below) put(int(at.id), row_dot(t, at, x));
        }
    }
    // in + sum G[j] in (a binomial pass or its transpose)
    template <class Pass, class Group, class Put>
    SMRT_HD static void pass(const Pass &t, const Group &g, const double *G, const double *in, Put &&put) {
        for (int r = g.lane; r < Pass::kRows; r += Group::G) {
            const RowAt at = t.at[r];
            const int b = at.beg;
            put(int(at.id), dot(at.len, in[at.id], [&](int i, double &v, double &y) {
                    y = in[t.col[b + i]];
                    v = G[t.j[b + i]];
                }));
        }
        g.sync();
    }
    template <class Pass, class Group>
    SMRT_HD static void pass(const Pass &t, const Group &g, const double *G, const double *in, double *out) {
        pass(t, g, G, in, [&](int p, double v) { out[p] = v; });
    }
    SMRT_HD double u_of(int k) const { return k == 0 ? u[0] : (k == 1 ? u[1] : u[2]); }
    SMRT_HD static double *g_of(double *V, int sign, int k) { return V + oG + (3 * sign + k) * (N + 1); }
    SMRT_HD static double inv_of(int j) { return j == 1 ? 1.0 : (j == 2 ? 0.5 : (j == 3 ? 1.0 / 3.0 : (j == 4 ? 0.25 : 0.2))); }
    // z_p = C[n][1] a_p + C[n][2] (t b)_p, n the order of p + 2 (t: del or trT)
    template <class Rows, class Group>
    SMRT_HD static void lift(const Tab &tab, const Rows &t, const Group &g, const double *a, const double *b,
                             const double *C, double *z) {
        for (int p = g.lane; p < M2; p += Group::G) {
            const int o = tab.ord[p];
            double v = C[Tab::c_slot(o + 2, 1)] * a[p];
            if (N >= 4 && o >= 2) {
                v = fma(C[Tab::c_slot(o + 2, 2)], row_dot(t, t.at[t.row[p]], b), v);
            }
            z[p] = v;
        }
        g.sync();
    }

    // F2: rho, u, theta and its powers from the raw moments; true when rho and theta are positive
    SMRT_HD bool conserved(double *V) {
        const double *Rc = V + oRc;
        rhom1 = Rc[0];
        rho = 1.0 + rhom1;
        ir = 1.0 / rho;
        u[0] = Rc[mi_pos(1, 0, 0)] * ir;
        u[1] = Rc[mi_pos(0, 1, 0)] * ir;
        u[2] = Rc[mi_pos(0, 0, 1)] * ir;
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        thm1 = (Rc[mi_pos(2, 0, 0)] + Rc[mi_pos(0, 2, 0)] + Rc[mi_pos(0, 0, 2)] - 3.0 * rhom1 - rho * uu) * ir *
               (1.0 / 3.0);
        th = 1.0 + thm1;
#ifdef __CUDA_ARCH__
        const double is = rsqrt(th);
#else
        const double is = 1.0 / sqrt(th);
#endif
        const double sq = th * is;
        double a = 1.0, b = 1.0;
        for (int j = 0; j <= N; ++j) {  // every lane writes the same values
            V[oPw + j] = a;
            V[oPw + N + 1 + j] = b;
            a *= is;
            b *= sq;
        }
        return rho > 0.0 && th > 0.0;
    }

    // F2 - F4: V's raw moments to the local-frame coefficients td; G of both transforms. False when
    // rho or theta is not positive.
    template <class Group>
    SMRT_HD bool local(const Tab &t, const Group &g, double *V) {
        const bool ok = conserved(V);
        rows(t.hd, g, V + oRc, [&](int a, double v) { V[oTa + a] = a == 0 ? rho : v; });
        for (int r = g.lane; r < 6; r += Group::G) {
            const double uk = r < 3 ? -u_of(r) : u_of(r - 3), t1 = r < 3 ? -thm1 : thm1;
            double *G = V + oG + r * (N + 1);
            double a = 1.0, b = uk;
            G[0] = a;
            G[1] = b;
            for (int j = 1; j < N; ++j) {
                const double n = (uk * b + t1 * a) * inv_of(j + 1);
                G[j + 1] = n;
                a = b;
                b = n;
            }
        }
        g.sync();
        pass(t.pass[0], g, g_of(V, 0, 0), V + oTa, V + oP1);
        pass(t.pass[1], g, g_of(V, 0, 1), V + oP1, V + oP2);
        pass(t.pass[2], g, g_of(V, 0, 2), V + oP2, [&](int p, double v) { V[oTd + p] = v * V[oPw + t.ord[p]]; });
        return ok;
    }

    // F2 - F6: V's raw moments to td, td', y, q1, q2 (F6's last pass is left to the callers).
    // model 1: ES-BGK with parameter es_b. False when rho or theta is not positive.
    template <class Group>
    SMRT_HD bool forward(const Tab &t, const Group &g, double *V, const double *tauA, const double *tauB, int model,
                         double es_b) {
        const bool ok = local(t, g, V);
        for (int k = g.lane; k < KT; k += Group::G) {  // the relaxation factors
            const double R = 1.0 / fma(tauB[k], rho, tauA[k]);
            V[oS + KT + k] = R;
            V[oS + k] = 1.0 - rho * R;
        }
        g.sync();
        rows(t.cj, g, V + oS, [&](int c, double v) { V[oC + c] = v; });
        g.sync();
        // F5
        if (model == 1) {
            const double tau = fma(tauB[0], rho, tauA[0]) * ir, om = 1.0 / tau;
            const double bp = 1.0 - (1.0 - es_b) * tau / fma(-0.5, es_b, tau);
            const double s = 1.0 - om, s2 = fma(om, bp, s), k4 = om * bp * bp * 0.5 * ir;
            for (int p = g.lane; p < M; p += Group::G) {
                const int n = t.ord[p];
                double v = V[oTd + p] * (n == 2 ? s2 : s);
                if (n == 4) {
                    double t4 = 0.0;
                    for (int i = 0; i < t.es_n[p]; ++i) t4 = fma(V[oTd + t.es_q1[p][i]], V[oTd + t.es_q2[p][i]], t4);
                    v = fma(k4, t4, v);
                }
                put_y(t, V, p, v);
            }
            g.sync();
        } else {
            // t1 = tr td, t2 = tr t1, z = C1 t1 + C2 delta t2, td' = C0 td + delta z
            rows(t.tr, g, V + oTd, [&](int p, double v) { V[oT1 + p] = v; });
            g.sync();
            if constexpr (N >= 4) {
                rows(t.tr, g, V + oT1, [&](int p, double v) { V[oT2 + p] = v; }, M4);
                g.sync();
            }
            lift(t, t.del, g, V + oT1, V + oT2, V + oC, V + oZ);
            rows(t.del, g, V + oZ, [&](int p, double v) {
                const int o = t.ord[p];
                put_y(t, V, p, o < 2 ? 0.0 : fma(V[oC + Tab::c_slot(o, 0)], V[oTd + p], v));
            });
            g.sync();
        }
        // F6
        pass(t.pass[0], g, g_of(V, 1, 0), V + oY, V + oQ1);
        pass(t.pass[1], g, g_of(V, 1, 1), V + oQ1, V + oQ2);
        return ok;
    }
    SMRT_HD void put_y(const Tab &t, double *V, int p, double v) const {
        const int o = t.ord[p];
        V[oTdp + p] = v;
        V[oY + p] = o == 0 ? rho : (o == 1 ? 0.0 : v * V[oPw + N + 1 + o]);
    }

    // The collision: V's raw moments (c-scaled) -> rebuild coefficients before their c^|g| scaling,
    // handed to put(g, value)
    template <class Group, class Put>
    SMRT_HD bool collide(const Tab &t, const Group &g, double *V, const double *tauA, const double *tauB, int model,
                         double es_b, Put &&put) {
        const bool ok = forward(t, g, V, tauA, tauB, model, es_b);
        pass(t.pass[2], g, g_of(V, 1, 2), V + oQ2, [&](int p, double v) { V[oP1 + p] = p == 0 ? rhom1 : v; });
        rows(t.hfT, g, V + oP1, put);
        g.sync();
        return ok;
    }

    // The adjoint (stages F7' .. F2' of adjoint.cuh): V's raw moments and Lc (c-scaled) -> the raw
    // moments' adjoint, handed to put(g, value); V + oTau: lam . d out / d tau_c,k.
    template <class Group, class Put>
    SMRT_HD void adjoint(const Tab &t, const Group &g, double *V, const double *tauA, const double *tauB, double dAdt,
                         double dBdt, Put &&put) {
        forward(t, g, V, tauA, tauB, 0, 0.0);
        // F7', F6'
        double tap0 = 0.0;
        rows(t.hf, g, V + oLc, [&](int a, double v) { V[oTapb + a] = v; });
        g.sync();
        tap0 = V[oTapb];
        g.sync();
        if (g.lane == 0) V[oTapb] = 0.0;  // ta'_0 := rho - 1 after the transform
        g.sync();
        pass(t.passT[2], g, g_of(V, 1, 2), V + oTapb, V + oQ2b);
        pass(t.passT[1], g, g_of(V, 1, 1), V + oQ2b, V + oQ1b);
        pass(t.passT[0], g, g_of(V, 1, 0), V + oQ1b, [&](int p, double v) {
            const int o = t.ord[p];
            V[oYb + p] = v;
            V[oTdpb + p] = o < 2 ? 0.0 : v * V[oPw + N + 1 + o];
        });
        // F5': w1 = delta^T tdpb, w2 = delta^T w1, x1 = C1 w1 + C2 tr^T w2, tdb = C0 tdpb + tr^T x1
        rows(t.delT, g, V + oTdpb, [&](int p, double v) { V[oW1 + p] = v; });
        g.sync();
        if constexpr (N >= 4) {
            rows(t.delT, g, V + oW1, [&](int p, double v) { V[oW2 + p] = v; }, M4);
            g.sync();
        }
        lift(t, t.trT, g, V + oW1, V + oW2, V + oC, V + oX1);
        rows(t.trT, g, V + oX1, [&](int p, double v) {
            const int o = t.ord[p];
            const double b = o < 2 ? 0.0 : fma(V[oC + Tab::c_slot(o, 0)], V[oTdpb + p], v);
            V[oTdb + p] = b;
            V[oP3b + p] = o < 2 ? 0.0 : b * V[oPw + o];
        });
        g.sync();
        // F4'
        pass(t.passT[2], g, g_of(V, 0, 2), V + oP3b, V + oP2b);
        pass(t.passT[1], g, g_of(V, 0, 1), V + oP2b, V + oP1b);
        pass(t.passT[0], g, g_of(V, 0, 0), V + oP1b, V + oTab);
        // sums: the adjoints of G (6 N sums over pairs of slots, longest first), of C, and the two
        // theta sums per order
        constexpr int kGs = 6 * N, kDots = 5 * (N - 1);
        for (int r = g.lane; r < kGs + kDots; r += Group::G) {
            if (r < kGs) {
                const int j = r / 6 + 1, sk = r % 6, k = sk % 3;
                const int oo = sk < 3 ? (k == 0 ? oP1b : (k == 1 ? oP2b : oP3b)) : (k == 0 ? oQ1b : (k == 1 ? oQ2b : oTapb));
                const int oi = sk < 3 ? (k == 0 ? oTa : (k == 1 ? oP1 : oP2)) : (k == 0 ? oY : (k == 1 ? oQ1 : oQ2));
                const double *a = V + oo, *b = V + oi;
                const int s = t.gbeg[j];
                V[oGb + sk * (N + 1) + j] = dot(t.gbeg[j + 1] - s, 0.0, [&](int i, double &v, double &y) {
                    v = a[t.gp[k][s + i]];
                    y = b[t.gq[k][s + i]];
                });
            } else {
                const int n = N - (r - kGs) / 5, what = (r - kGs) % 5;
                const int o = what == 3 ? n - 2 : (what == 4 ? n - 4 : n);
                if (o < 0) continue;
                const double *a = V + (what == 0 || what == 1 ? oTdpb : (what == 2 ? oTdb : (what == 3 ? oW1 : oW2)));
                const double *b = V + (what == 0 ? oTdp : (what <= 2 ? oTd : (what == 3 ? oT1 : oT2)));
                const int s = ord_off(o);
                const double acc = dot(ord_off(o + 1) - s, 0.0, [&](int i, double &v, double &y) {
                    v = a[s + i];
                    y = b[s + i];
                });
                V[what == 0 ? oA + n : (what == 2 ? oE + n : oCb + Tab::c_slot(n, what == 1 ? 0 : what - 2))] = acc;
            }
        }
        g.sync();
        for (int r = g.lane; r < 6; r += Group::G) {  // transposed recurrences of G
            const double uk = r < 3 ? -u_of(r) : u_of(r - 3), t1 = r < 3 ? -thm1 : thm1;
            const double *G = V + oG + r * (N + 1);
            double *Gb = V + oGb + r * (N + 1);
            double hi = Gb[N], lo = N > 1 ? Gb[N - 1] : 0.0, ub = 0.0, tb = 0.0;
            for (int j = N - 1; j >= 1; --j) {
                const double q = hi * inv_of(j + 1);
                ub = fma(q, G[j], ub);
                tb = fma(q, G[j - 1], tb);
                hi = fma(q, uk, lo);
                lo = j >= 2 ? fma(q, t1, Gb[j - 1 > 0 ? j - 1 : 0]) : 0.0;
            }
            V[oMx + 2 * r] = ub + hi;
            V[oMx + 2 * r + 1] = tb;
        }
        rows(t.cjT, g, V + oCb, [&](int k, double sb) {
            const double R = V[oS + KT + k];
            V[oSr + k] = -sb * tauA[k] * R * R;
            V[oTau + k] = sb * (rho * R * R * dAdt + rho * rho * R * R * dBdt);
        });
        g.sync();
        // F3', F2'
        const double *mx = V + oMx;
        double ub[3], tb = 0.0, rhob = tap0 + V[oYb] + V[oTab];
        for (int k = 0; k < 3; ++k) {
            ub[k] = mx[2 * (3 + k)] - mx[2 * k];
            tb += mx[2 * (3 + k) + 1] - mx[2 * k + 1];
        }
        double ts = 0.0;
        for (int n = 2; n <= N; ++n) ts = fma(0.5 * n, V[oA + n] - V[oE + n], ts);
        tb += ts / th;
        for (int k = 0; k < KT; ++k) rhob += V[oSr + k];
        const double t3 = tb * ir * (1.0 / 3.0);
        const double tab0 = V[oTab];
        rows(t.hdT, g, V + oTab, [&](int q, double v) {
            if (q == 0)  // slot 0 of ta is rho, not the transform of Rc
                v = v - tab0 + rhob - (ub[0] * u[0] + ub[1] * u[1] + ub[2] * u[2]) * ir + t3 * (uu - 3.0) - tb * thm1 * ir;
            else if (q <= 3)
                v += (q == 1 ? ub[0] : (q == 2 ? ub[1] : ub[2])) * ir - 2.0 * t3 * u_of(q - 1);
            else if (q == mi_pos(2, 0, 0) || q == mi_pos(0, 2, 0) || q == mi_pos(0, 0, 2))
                v += t3;
            put(q, v);
        });
        g.sync();
    }
};

// Population side: x (Q values, library order) to and from the transformed form of LaneOrbits.
template <class Lat, int N>
struct LanePops {
    using Tab = LaneOrbits<Lat, N>;
    template <class Group>
    SMRT_HD static void butterflies(const Tab &t, const Group &g, double *x) {
        for (int s = 0; s < 2; ++s) {
            const int n = s == 0 ? t.n0 : t.n1;
            for (int i = g.lane; i < 2 * n; i += Group::G) {
                const unsigned char *pr = s == 0 ? t.b0[i >> 1] : t.b1[i >> 1];
                double &a = x[2 * pr[0] + 1 + (i & 1)], &b = x[2 * pr[1] + 1 + (i & 1)];
                const double lo = a, hi = b;
                a = lo + hi;
                b = lo - hi;
            }
            g.sync();
        }
    }
    // populations -> pair sums and differences, transformed
    template <class Group>
    SMRT_HD static void analyse(const Tab &t, const Group &g, double *x) {
        for (int p = g.lane; p < Lat::NP; p += Group::G) {
            const double a = x[2 * p + 1], b = x[2 * p + 2];
            x[2 * p + 1] = a + b;
            x[2 * p + 2] = t.flip[p] ? b - a : a - b;
        }
        g.sync();
        butterflies(t, g, x);
    }
    // transformed even and odd parts -> values at the populations
    template <class Group, class Put>
    SMRT_HD static void synthesise(const Tab &t, const Group &g, double *x, Put &&put) {
        butterflies(t, g, x);
        for (int p = g.lane; p < Lat::NP; p += Group::G) {
            const double e = x[2 * p + 1], o = t.flip[p] ? -x[2 * p + 2] : x[2 * p + 2];
            put(2 * p + 1, e + o);
            put(2 * p + 2, e - o);
        }
        if (g.lane == 0) put(0, x[0]);
    }
};

}  // namespace smrt
