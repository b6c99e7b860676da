// Host harness for the fixed-point operator (fix_core.cuh) with an exponent per
// component and for the constant modes, as apply_fix.cu stages them; compiled by
// tests/test_fix_parts.py.  Returns 3 where a value lies outside the fixed-point range.
#include <vector>

#include "../paper_1607_03777_gb300/csrc/fix_core.cuh"

using namespace sip::fix;

namespace {

int biased(double v) { return int(bits_of(v) >> 52) & 0x7ff; }

template <int N, int TW, int TH>
int apply(int nx, int ny, double lx, double ly, const int* bc, double ch, const double* x, const double* eta,
          double* y) {
    using L = Tile<N, TW, TH>;
    const Scal k = make_scal<N>((ly / ny) / (lx / nx), ch);
    if (!k.ok) return 1;
    double ss[36];
    for (int q = 0; q < N * N; ++q) ss[q] = leg(q % N) * leg(q / N);
    std::vector<i64> buf((L::BYTES + 7) / 8, 0x5a5a5a5a5a5a5a5aLL);
    i64* sm = buf.data();
    double* seta = reinterpret_cast<double*>(sm + L::O_ETA);
    int* se = reinterpret_cast<int*>(sm + L::O_E);
    for (int ey0 = 0; ey0 < ny; ey0 += TH)
        for (int ex0 = 0; ex0 < nx; ex0 += TW) {
            const Mesh g{nx, ny, ex0, ey0, {bc[0], bc[1], bc[2], bc[3]}};
            for (int s = 0; s < L::NS; ++s) {
                int ex, ey, e[2] = {0, 0}, above[2];
                const bool in = staged_at<N, TW, TH>(g, s, ex, ey);
                const double* u = x + (in ? size_t(ey) * nx + ex : 0) * L::NB;
                for (int q = 0; in && q < L::NB; ++q)
                    if (q % L::NN) e[q / L::NN] = imax(e[q / L::NN], biased(u[q]));
                seta[s] = in ? eta[size_t(ey) * nx + ex] : 1.0;
                se[s] = expo_pack(e[0], e[1]);
                for (int q = 0; q < L::NB; ++q) {
                    const int c = q / L::NN, g1 = !in ? 0 : (q % L::NN ? e[c] : biased(u[q]));
                    if (g1 && (g1 < E_MIN || g1 > E_MAX)) return 3;
                    if (q % L::NN == 0) above[c] = g1 - e[c];
                    sm[s * L::XS + q] = g1 ? to_int(u[q] * in_factor<N>(ss[q % L::NN], g1)) : 0;
                }
                sm[s * L::XS + L::NB] = mean_pack(above[0], above[1]);
            }
            for (int t = 0; t < L::NT; ++t) phase_traces<N, TW, TH>(t, g, sm);
            for (int t = 0; t < L::NT; ++t) phase_lines<N, TW, TH, 0>(t, g, k, ss, sm);
            for (int t = 0; t < L::NT; ++t) phase_lines<N, TW, TH, 1>(t, g, k, ss, sm);
            for (int el = 0; el < L::NEL; ++el) {
                int ex, ey;
                if (!staged_at<N, TW, TH>(g, el, ex, ey)) continue;
                for (int q = 0; q < L::NB; ++q)
                    y[(size_t(ey) * nx + ex) * L::NB + q] = of_bits(sm[L::O_W + q * L::EP + el]);
            }
        }
    return 0;
}

}  // namespace

extern "C" int fix_apply_parts(int N, int nx, int ny, double lx, double ly, const int* bc, double ch,
                               const double* x, const double* eta, double* y) {
    switch (N) {
        case 2: return apply<2, 16, 8>(nx, ny, lx, ly, bc, ch, x, eta, y);
        case 3: return apply<3, 8, 8>(nx, ny, lx, ly, bc, ch, x, eta, y);
        case 4: return apply<4, 8, 4>(nx, ny, lx, ly, bc, ch, x, eta, y);
        case 5: return apply<5, 16, 2>(nx, ny, lx, ly, bc, ch, x, eta, y);
        case 6: return apply<6, 8, 4>(nx, ny, lx, ly, bc, ch, x, eta, y);
    }
    return 2;
}
