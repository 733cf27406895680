// lane_kernels.cuh -- the step and its adjoint on small batches of 1D lines, one cell per group of
// lanes (lane_cell.cuh says why). A block of 128 threads takes 128 / G consecutive cells of one
// line: it pulls their populations into shared memory together (consecutive cells of a plane side
// by side), each group runs its cell, and the block stores the results together.
//
// G = 32 (a cell per warp) or 16 (two). N = 4 has 35 moments: 32 lanes take 2 rounds per stage for
// one cell, 16 lanes 3 rounds for two. The larger group has the shorter chain, the smaller one does
// less work per cell.
#pragma once

#include "adjoint_kernels.cuh"
#include "kernels.cuh"
#include "lane_cell.cuh"

namespace smrt {

static __device__ const LaneMoments<3> kLaneMoments3 = LaneMoments<3>();
static __device__ const LaneMoments<4> kLaneMoments4 = LaneMoments<4>();
static __device__ const LaneMoments<5> kLaneMoments5 = LaneMoments<5>();
static __device__ const LaneOrbits<D3Q39, 3> kLaneOrbits39 = LaneOrbits<D3Q39, 3>();
static __device__ const LaneOrbits<D3Q103, 3> kLaneOrbits103n3 = LaneOrbits<D3Q103, 3>();
static __device__ const LaneOrbits<D3Q103, 4> kLaneOrbits103n4 = LaneOrbits<D3Q103, 4>();
template <int N>
SMRT_D const LaneMoments<N> &lane_moments();
template <>
SMRT_D const LaneMoments<3> &lane_moments<3>() { return kLaneMoments3; }
template <>
SMRT_D const LaneMoments<4> &lane_moments<4>() { return kLaneMoments4; }
template <>
SMRT_D const LaneMoments<5> &lane_moments<5>() { return kLaneMoments5; }
template <class Lat, int N>
SMRT_D const LaneOrbits<Lat, N> &lane_orbits();
template <>
SMRT_D const LaneOrbits<D3Q39, 3> &lane_orbits<D3Q39, 3>() { return kLaneOrbits39; }
template <>
SMRT_D const LaneOrbits<D3Q103, 3> &lane_orbits<D3Q103, 3>() { return kLaneOrbits103n3; }
template <>
SMRT_D const LaneOrbits<D3Q103, 4> &lane_orbits<D3Q103, 4>() { return kLaneOrbits103n4; }

constexpr int kLaneThreads = 128;

template <int LG>
struct LaneGroup {
    static constexpr int G = LG;
    static_assert(LG == 16 || LG == 32, "whole warps, one or two cells each");
    int lane;
    SMRT_D void sync() const { __syncwarp(); }  // all cells of a warp run every stage
};

// Shared memory of a block: the tables, then per cell V and the populations (X; the adjoint also
// keeps the weighted adjoint state, Y).
template <class Lat, int N, bool Adjoint, int G>
struct LaneShared {
    static constexpr int kCells = kLaneThreads / G;  // cells per block
    using C = LaneCell<N>;
    LaneMoments<N> m;
    LaneOrbits<Lat, N> o;
    double cp[(N + 2) / 2 * 2];                     // c^j
    double w[(Lat::NP + 2) / 2 * 2];                // weights: rest, then of each pair
    static constexpr int kV = Adjoint ? int(C::kAdjoint) : int(C::kForward);
    double V[kCells][kV];
    double X[kCells][Lat::Q];
    double Y[Adjoint ? kCells : 1][Lat::Q];
};

template <class Tab>
SMRT_D void lane_copy(Tab &dst, const Tab &src) {
    static_assert(sizeof(Tab) % 16 == 0, "copied 16 bytes at a time");
    const uint4 *s = reinterpret_cast<const uint4 *>(&src);
    uint4 *d = reinterpret_cast<uint4 *>(&dst);
    for (int i = threadIdx.x; i < int(sizeof(Tab) / 16); i += kLaneThreads) d[i] = s[i];
}

// The block's cells: x0 .. x0 + kCells - 1 of its tile's instance; bpt blocks per tile.
template <class Lat, int N, class T, bool FixedX, class Sh>
struct LaneBlock {
    static constexpr int kCells = Sh::kCells;
    const StepArgs<Lat, T> &a;
    Sh &s;
    const InstanceInfo &in;
    const int j, x0, L;
    const long long base;
    SMRT_D LaneBlock(const StepArgs<Lat, T> &a_, Sh &s_, int bpt)
        : a(a_), s(s_), in(a_.inst[a_.tiles[blockIdx.x / bpt].x]), j(a_.tiles[blockIdx.x / bpt].x),
          x0(a_.tiles[blockIdx.x / bpt].y + int(blockIdx.x % bpt) * kCells), L(in.nx), base(in.cell_off) {}
    // the tables and the cells' pulled populations (zero beyond the line's last cell)
    SMRT_D void load() {
        lane_copy(s.m, lane_moments<N>());
        lane_copy(s.o, lane_orbits<Lat, N>());
        if (threadIdx.x == 0) {
            s.cp[0] = 1.0;
            for (int k = 1; k <= N; ++k) s.cp[k] = s.cp[k - 1] * a.cd;
        }
        for (int p = threadIdx.x; p <= Lat::NP; p += kLaneThreads) s.w[p] = a.wpd[p];
        const T *gl = a.ghosts + (long long)j * 2 * Lat::Q;
        for (int q = threadIdx.x; q < Lat::Q * kCells; q += kLaneThreads) {
            const int i = q / kCells, c = q % kCells, x = x0 + c;
            double v = 0.0;
            if (x < L) {
                const int xs = x - (lane_orbits<Lat, N>().ex[i] + in.kx);
                if (FixedX && xs < 0)
                    v = double(gl[i]);
                else if (FixedX && xs >= L)
                    v = double(gl[Lat::Q + i]);
                else
                    v = double(a.fin[a.plane[i] + base + wrap(xs, L)]);
            }
            s.X[c][i] = v;
        }
    }
    // c-scaled raw moments of x into R
    template <class Group>
    SMRT_D void moments(const Group &g, double *x, double *R) {
        LanePops<Lat, N>::analyse(s.o, g, x);
        LaneCell<N>::rows(s.o.raw, g, x, [&](int k, double v) { R[k] = v * s.cp[s.m.ord[k]]; });
    }
};

template <class Lat, int N, bool FixedX, int G>
__global__ void __launch_bounds__(kLaneThreads) step_lane_kernel(StepArgs<Lat, double> a, int bpt) {
    extern __shared__ __align__(128) unsigned char dyn[];
    using Sh = LaneShared<Lat, N, false, G>;
    constexpr int kCells = Sh::kCells;
    Sh &s = *reinterpret_cast<Sh *>(dyn);
    LaneBlock<Lat, N, double, FixedX, Sh> b(a, s, bpt);
    if (b.x0 >= b.L) return;  // the whole block
    b.load();
    __syncthreads();
    const LaneGroup<G> g{int(threadIdx.x) % G};
    const int c = int(threadIdx.x) / G;
    double *V = s.V[c], *x = s.X[c], *P = V + LaneCell<N>::oTa;
    b.moments(g, x, V + LaneCell<N>::oRc);
    g.sync();
    LaneCell<N> cell;
    const bool ok = cell.collide(s.m, g, V, b.in.tauA, b.in.tauB, b.in.model, b.in.es_b,
                                 [&](int k, double v) { P[k] = v * s.cp[s.m.ord[k]]; });
    if (!ok && g.lane == 0 && b.x0 + c < b.L) atomicOr(a.health, 1u);
    LaneCell<N>::rows(s.o.rawT, g, P, [&](int i, double v) { x[i] = v; });
    g.sync();
    LanePops<Lat, N>::synthesise(s.o, g, x, [&](int i, double v) { x[i] = s.w[(i + 1) >> 1] * v; });
    __syncthreads();
    for (int q = threadIdx.x; q < Lat::Q * kCells; q += kLaneThreads) {
        const int i = q / kCells, cc = q % kCells;
        if (b.x0 + cc < b.L) a.fout[a.plane[i] + b.base + b.x0 + cc] = s.X[cc][i];
    }
}

// partials[block][tau]: the block's cells in order
template <class Lat, int N, class T, bool FixedX, int G>
__global__ void __launch_bounds__(kLaneThreads) adjoint_lane_kernel(StepArgs<Lat, T> a, const double *lam_in,
                                                                    double *lam_out, double *partials, int bpt) {
    constexpr int KT = ntau(N);
    extern __shared__ __align__(128) unsigned char dyn[];
    using Sh = LaneShared<Lat, N, true, G>;
    constexpr int kCells = Sh::kCells;
    using C = LaneCell<N>;
    Sh &s = *reinterpret_cast<Sh *>(dyn);
    LaneBlock<Lat, N, T, FixedX, Sh> b(a, s, bpt);
    if (b.x0 >= b.L) {
        if (threadIdx.x < KT) partials[(long long)blockIdx.x * KT + threadIdx.x] = 0.0;
        return;
    }
    b.load();
    for (int q = threadIdx.x; q < Lat::Q * kCells; q += kLaneThreads) {
        const int i = q / kCells, cc = q % kCells;
        s.Y[cc][i] = b.x0 + cc < b.L ? a.wpd[(i + 1) >> 1] * lam_in[a.plane[i] + b.base + b.x0 + cc] : 0.0;
    }
    __syncthreads();
    const LaneGroup<G> g{int(threadIdx.x) % G};
    const int c = int(threadIdx.x) / G;
    double *V = s.V[c], *x = s.X[c], *P = V + C::oLc;
    b.moments(g, x, V + C::oRc);
    b.moments(g, s.Y[c], V + C::oLc);
    g.sync();
    C cell;
    cell.adjoint(s.m, g, V, b.in.tauA, b.in.tauB, b.in.dAdt, b.in.dBdt,
                 [&](int k, double v) { P[k] = v * s.cp[s.m.ord[k]]; });
    C::rows(s.o.rawT, g, P, [&](int i, double v) { x[i] = v; });
    g.sync();
    LanePops<Lat, N>::synthesise(s.o, g, x, [&](int i, double v) { x[i] = v; });
    __syncthreads();
    // the streaming's transpose: lam_i at the cell population i was pulled from; zero at (i, x)
    // when no cell pulls population i from x
    for (int q = threadIdx.x; q < Lat::Q * kCells; q += kLaneThreads) {
        const int i = q / kCells, cc = q % kCells, xc = b.x0 + cc;
        if (xc >= b.L) continue;
        const int sx = s.o.ex[i] + b.in.kx, xs = xc - sx, xd = xc + sx;
        double *o = lam_out + a.plane[i] + b.base;
        if (!FixedX)
            o[wrap(xs, b.L)] = s.X[cc][i];
        else if (xs >= 0 && xs < b.L)
            o[xs] = s.X[cc][i];
        if (FixedX && (xd < 0 || xd >= b.L)) o[xc] = 0.0;
    }
    if (threadIdx.x < KT) {
        double acc = 0.0;
        for (int cc = 0; cc < kCells && b.x0 + cc < b.L; ++cc) acc += s.V[cc][C::oTau + threadIdx.x];
        partials[(long long)blockIdx.x * KT + threadIdx.x] = acc;
    }
}

}  // namespace smrt
