// Host harness for the fixed-point operator (fix_core.cuh), compiled by
// tests/test_fix_host.py: the kernel's phases run tile by tile on the host.
#include <vector>

#include "../paper_1607_03777_gb300/csrc/fix_core.cuh"

using namespace sip::fix;

namespace {

template <int N, int TW, int TH>
int apply(int nx, int ny, double lx, double ly, const int* bc, double ch, const double* x, const double* eta,
          double* y) {
    using L = Tile<N, TW, TH>;
    const Scal k = make_scal<N>((ly / ny) / (lx / nx), ch);
    if (!k.ok) return 1;
    double ss[36];
    for (int q = 0; q < N * N; ++q) ss[q] = leg(q % N) * leg(q / N);
    std::vector<i64> buf((L::BYTES + 7) / 8);
    i64* sm = buf.data();
    double* seta = reinterpret_cast<double*>(sm + L::O_ETA);
    int* se = reinterpret_cast<int*>(sm + L::O_E);
    for (int ey0 = 0; ey0 < ny; ey0 += TH)
        for (int ex0 = 0; ex0 < nx; ex0 += TW) {
            const Mesh g{nx, ny, ex0, ey0, {bc[0], bc[1], bc[2], bc[3]}};
            for (int s = 0; s < L::NS; ++s) {
                int ex, ey, e = 0;
                const bool in = staged_at<N, TW, TH>(g, s, ex, ey);
                const double* u = x + (in ? size_t(ey) * nx + ex : 0) * L::NB;
                for (int q = 0; in && q < L::NB; ++q) {
                    const int b = int(bits_of(u[q]) >> 52) & 0x7ff;
                    e = b > e ? b : e;
                }
                seta[s] = in ? eta[size_t(ey) * nx + ex] : 1.0;
                se[s] = e;
                for (int q = 0; q < L::NB; ++q)
                    sm[s * L::XS + q] = e ? to_int(u[q] * in_factor<N>(ss[q % (N * N)], e)) : 0;
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

extern "C" int fix_apply(int N, int nx, int ny, double lx, double ly, const int* bc, double ch,
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
