// Host build of the group-of-lanes collision and adjoint (csrc/lane_cell.cuh) with a group of one
// lane, beside the one-thread adjoint (csrc/adjoint.cuh), for a CPU test. Library order.
#include "../../paper_2401_11086_gb300/csrc/adjoint.cuh"
#include "../../paper_2401_11086_gb300/csrc/lane_cell.cuh"

using namespace smrt;

struct OneLane {
    static constexpr int G = 1;
    int lane = 0;
    SMRT_HD void sync() const {}
};

template <class Lat, int N>
static void raw(const LaneOrbits<Lat, N> &t, double *x, double c, double *R) {
    const OneLane g;
    LanePops<Lat, N>::analyse(t, g, x);
    LaneCell<N>::rows(t.raw, g, x, [&](int k, double v) {
        for (int j = 0; j < mi_order(k); ++j) v *= c;
        R[k] = v;
    });
}
template <class Lat, int N, class Put>
static void back(const LaneOrbits<Lat, N> &t, const double *P, double c, Put &&put) {
    const OneLane g;
    double sc[nmom(N)], x[Lat::Q];
    for (int k = 0; k < nmom(N); ++k) {
        sc[k] = P[k];
        for (int j = 0; j < mi_order(k); ++j) sc[k] *= c;
    }
    LaneCell<N>::rows(t.rawT, g, sc, [&](int i, double v) { x[i] = v; });
    LanePops<Lat, N>::synthesise(t, g, x, put);
}

template <class Lat, int N>
static void step(const double *f, double c, const double *wp, const double *tauA, const double *tauB, int model,
                 double es_b, double *out) {
    using C = LaneCell<N>;
    static const LaneMoments<N> tm;
    static const LaneOrbits<Lat, N> to;
    double V[C::kForward], x[Lat::Q], P[nmom(N)];
    for (int i = 0; i < Lat::Q; ++i) x[i] = f[i];
    raw<Lat, N>(to, x, c, V + C::oRc);
    C cell;
    cell.collide(tm, OneLane(), V, tauA, tauB, model, es_b, [&](int k, double v) { P[k] = v; });
    back<Lat, N>(to, P, c, [&](int i, double v) { out[i] = wp[(i + 1) / 2] * v; });
}

template <class Lat, int N>
static void vjp(const double *f, const double *lam, double c, const double *wp, const double *tauA, const double *tauB,
                double dAdt, double dBdt, double *fb, double *taub) {
    using C = LaneCell<N>;
    static const LaneMoments<N> tm;
    static const LaneOrbits<Lat, N> to;
    double V[C::kAdjoint], x[Lat::Q], P[nmom(N)];
    for (int i = 0; i < Lat::Q; ++i) x[i] = f[i];
    raw<Lat, N>(to, x, c, V + C::oRc);
    for (int i = 0; i < Lat::Q; ++i) x[i] = wp[(i + 1) / 2] * lam[i];
    raw<Lat, N>(to, x, c, V + C::oLc);
    C cell;
    cell.adjoint(tm, OneLane(), V, tauA, tauB, dAdt, dBdt, [&](int k, double v) { P[k] = v; });
    back<Lat, N>(to, P, c, [&](int i, double v) { fb[i] = v; });
    for (int k = 0; k < ntau(N); ++k) taub[k] = V[C::oTau + k];
}

template <class Lat, int N>
static void vjp_thread(const double *f, const double *lam, double c, const double *wp, const double *tauA,
                       const double *tauB, double dAdt, double dBdt, double *fb, double *taub) {
    double ff[Lat::Q], ll[Lat::Q], ww[Lat::NP + 1], out[Lat::Q], tb[ntau(N)];
    for (int i = 0; i < Lat::Q; ++i) ff[i] = f[i], ll[i] = lam[i];
    for (int p = 0; p <= Lat::NP; ++p) ww[p] = wp[p];
    for (int k = 0; k < ntau(N); ++k) tb[k] = 0.0;
    collide_vjp<Lat, N>(ff, ll, c, ww, tauA, tauB, dAdt, dBdt, out, tb);
    for (int i = 0; i < Lat::Q; ++i) fb[i] = out[i];
    for (int k = 0; k < ntau(N); ++k) taub[k] = tb[k];
}

#define SET(tag, Lat, N)                                                                                          \
    void step_##tag(const double *f, double c, const double *wp, const double *A, const double *B, int m, double b, \
                    double *o) {                                                                                  \
        step<Lat, N>(f, c, wp, A, B, m, b, o);                                                                    \
    }                                                                                                             \
    void vjp_##tag(const double *f, const double *l, double c, const double *wp, const double *A, const double *B,  \
                   double da, double db, double *fb, double *tb) {                                                \
        vjp<Lat, N>(f, l, c, wp, A, B, da, db, fb, tb);                                                           \
    }                                                                                                             \
    void vjpt_##tag(const double *f, const double *l, double c, const double *wp, const double *A, const double *B, \
                    double da, double db, double *fb, double *tb) {                                               \
        vjp_thread<Lat, N>(f, l, c, wp, A, B, da, db, fb, tb);                                                    \
    }

extern "C" {
SET(d3q39_n3, D3Q39, 3)
SET(d3q103_n3, D3Q103, 3)
SET(d3q103_n4, D3Q103, 4)
}
