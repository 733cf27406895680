// Host build of the run-time orbit rows (csrc/lattices.cuh) that the split-precision step loops
// over, for a CPU test of what they hold.
#include "../../paper_2401_11086_gb300/csrc/lattices.cuh"

using namespace smrt;

// Per row: mask, np, then per member (v, population of v, of -v, their staged offsets), 7 ints;
// mono and cls: per row and slot of order <= N, a^gamma (0 when the slot vanishes on the mask) and
// the transform entry. Returns the number of rows; *seg: elements per staged row.
template <class Lat>
static int dump(int N, int *rows, int *mono, int *cls, int *seg) {
    constexpr OrbitRows<Lat> R{};
    const int M = nmom(N);
    *seg = staged_row<Lat>();
    for (int mask = 1; mask < 8; ++mask)
        for (int o = R.first[mask]; o < R.first[mask + 1]; ++o) {
            int *q = rows + 30 * o;
            q[0] = mask;
            q[1] = 1 << (mask_axes(mask) - 1);
            for (int b = 0; b < q[1]; ++b) {
                int *m = q + 2 + 7 * b;
                for (int d = 0; d < 3; ++d) m[d] = R.row[o].e[b][d];
                m[3] = R.row[o].ip[b], m[4] = R.row[o].im[b];
                m[5] = R.row[o].sp[b], m[6] = R.row[o].sm[b];
            }
            for (int g = 0; g < M; ++g) {
                mono[o * M + g] = mask_has(mask, g) ? R.row[o].mono[g] : 0;
                cls[o * M + g] = mask_class(mask, g);
            }
        }
    return R.first[8];
}

extern "C" {
int rows_d3q39(int N, int *r, int *m, int *c, int *s) { return dump<D3Q39>(N, r, m, c, s); }
int rows_d3q103(int N, int *r, int *m, int *c, int *s) { return dump<D3Q103>(N, r, m, c, s); }
void slot_components(int N, int *out) {
    for (int g = 0; g < nmom(N); ++g)
        for (int d = 0; d < 3; ++d) out[3 * g + d] = mi_comp(g, d);
}
}
