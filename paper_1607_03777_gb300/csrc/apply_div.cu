// B and B^T in FP64 (eq. divergence_form): b_h(v, q) = -int q div v + int {q} [[v.n]].
//
// What bounds them: the FP64 pipe.  One thread per mode (the double-double
// kernels of apply.cu) recomputes each face trace for every mode along the
// normal and multiplies the zeros of the 1D tables; one thread per (element,
// line) forms a line's scaled entries, their even and odd sums (both end
// traces) and their prefix sums (int l_p l_q' = 2 l_p(1) l_q(1) for q > p, q - p
// odd) once: 37 (B) and 41 (B^T) FP64 operations per line at k = 4 instead of 230, and
// the FP64 pipe 84 and 80 % busy (512^2).
// 250 x 190, k = 4, both operators: 417 us before, 72 now.
//
// Mode q receives (h / 2) l_q(1) (f_1 - (-1)^q f_0 - 2 sum of the other parity beyond q) with
// f_s = c_s own_s + neighbour_s / 2 and own_s = even +- odd sum.  In the traces' sum and
// difference one parity cancels between the faces, so its coefficients c_1 +- c_0 are
// formed first; with the sums by fused multiply-adds the error is below that of the
// one-thread-per-mode kernels (the difference of rounded traces was above it).
//
// Layout: a CTA serves 32 elements of one mesh row, a warp per line, a lane per
// element.  The row, its left and right neighbour and the rows below and above
// are read with consecutive lanes on consecutive entries and kept in shared
// memory with an odd element stride; results go back the same way.
#include "sip_elem.cuh"
#include "sip_internal.h"

namespace sip {

namespace {

constexpr int WX = 32;   // elements per CTA

// sqrt(2 i + 1) = sqrt(2) l_i(1): without rounding for i = 0 and 4
__device__ constexpr double kRoot[7] = {1.0, 1.7320508075688772, 2.23606797749979, 2.6457513110645907, 3.0,
                             3.3166247903554, 3.605551275463989};

struct DivArgs {
    const double* in;
    double* out;
    int nx, ny;
    int bc[4];
    double hl[2][7];   // sqrt(2 q + 1) times a quarter of the face's length, per direction of the normal
};

// Rows ey - 1, ey, ey + 1 of a vector of NE entries per element, columns
// ex0 - 1 .. ex0 + 32, into s[row][column][entry]; entries outside the mesh are left
// unset and must not be read.
template <int NE, int ES>
__device__ __forceinline__ void load_rows(const DivArgs& a, int ex0, int ey, double* s) {
    const int lo = max(ex0 - 1, 0), hi = min(ex0 + WX + 1, a.nx);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int y = ey + r - 1;
        double* d = s + (r * (WX + 2) + lo - (ex0 - 1)) * ES;
        if (y < 0 || y >= a.ny) continue;
        const double* g = a.in + (size_t(y) * a.nx + lo) * NE;
        const int n = (hi - lo) * NE;
#pragma unroll 4
        for (int q = threadIdx.x; q < n; q += blockDim.x) d[(q / NE) * ES + q % NE] = g[q];
    }
}

// Weighted even and odd sums of a line: traces at the ends are ev + od, ev - od.
template <int L>
__device__ __forceinline__ void even_odd(const double* p, int stride, double& ev, double& od) {
    ev = od = 0.0;
#pragma unroll
    for (int i = 0; i < L; ++i) {
        double& a = i % 2 == 0 ? ev : od;
        a = fma(kRoot[i], p[i * stride], a);
    }
}

// What a line's traces give to the modes of either parity (even: difference of the ends,
// odd: sum), sg / 2 the neighbours' weight; nb entries to the neighbour on the plus side.
template <int L>
__device__ __forceinline__ void end_traces(const DivArgs& a, int dir, int ex, int ey, const double* p, int stride,
                                           int nb, double sg, double& fe, double& fo) {
    double ev, od, e2, o2, c[2], n[2];
    even_odd<L>(p, stride, ev, od);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const bool in = dir == 0 ? (s ? ex < a.nx - 1 : ex > 0) : (s ? ey < a.ny - 1 : ey > 0);
        n[s] = 0.0;
        if (in) {
            even_odd<L>(p + (s ? nb : -nb), stride, e2, o2);
            n[s] = s ? e2 - o2 : e2 + o2;
        }
        c[s] = in ? 0.5 : (a.bc[2 * dir + s] == SIP_BC_NEUMANN ? 0.0 : 1.0);
    }
    const double cp = c[1] + c[0], cm = c[1] - c[0];
    fe = fma(sg, n[1] - n[0], fma(cm, ev, cp * od));
    fo = fma(sg, n[1] + n[0], fma(cm, od, cp * ev));
}

// B p: the N modes along the normal of line m (m < K) of component dir.
template <int N>
__global__ void __launch_bounds__(WX * 2 * (N - 1)) k_div_B(const DivArgs a) {
    grid_dep_wait();
    constexpr int K = N - 1, MP = K * K, ES = MP | 1, NN = N * N, NB = 2 * NN, OS = NB + 1;
    extern __shared__ double sm[];
    double* sp = sm;                        // [3][WX + 2][ES]
    double* so = sm + 3 * (WX + 2) * ES;    // [WX][OS]
    const int ntx = (a.nx + WX - 1) / WX, ex0 = int(blockIdx.x % ntx) * WX, ey = blockIdx.x / ntx;
    load_rows<MP, ES>(a, ex0, ey, sp);
    for (int q = threadIdx.x; q < WX * OS; q += blockDim.x) so[q] = 0.0;   // lines m = K stay zero
    __syncthreads();
    const int lane = threadIdx.x % 32, dir = (threadIdx.x / 32) / K, m = (threadIdx.x / 32) % K;
    const int ex = ex0 + lane;
    if (ex < a.nx) {
        const int stride = dir == 0 ? 1 : K, at = dir == 0 ? m * K : m;
        const double* p = sp + ((WX + 2) + lane + 1) * ES + at;
        const int nb = dir == 0 ? ES : (WX + 2) * ES;   // to the neighbour on the plus side
        double fe, fo;
        end_traces<K>(a, dir, ex, ey, p, stride, nb, 0.5, fe, fo);
        double* o = so + lane * OS + dir * NN + (dir == 0 ? m * N : m);
        double pe = 0.0, po = 0.0;   // sums of the even / odd entries below q
#pragma unroll
        for (int q = 0; q < N; ++q) {
            o[dir == 0 ? q : q * N] = a.hl[dir][q] * (q % 2 == 0 ? fma(-2.0, po, fe) : fma(-2.0, pe, fo));
            if (q < K) {
                double& b = q % 2 == 0 ? pe : po;
                b = fma(kRoot[q], p[q * stride], b);
            }
        }
    }
    __syncthreads();
    const int n = (min(ex0 + WX, a.nx) - ex0) * NB;
    double* g = a.out + (size_t(ey) * a.nx + ex0) * NB;
#pragma unroll 4
    for (int q = threadIdx.x; q < n; q += blockDim.x) g[q] = so[(q / NB) * OS + q % NB];
}

// B^T u: the K modes along the normal that line m (m < K) of component dir
// gives; columns (dir 1) add to what rows (dir 0) left.
template <int N>
__global__ void __launch_bounds__(WX * 2 * (N - 1)) k_div_Bt(const DivArgs a) {
    grid_dep_wait();
    constexpr int K = N - 1, MP = K * K, NN = N * N, NB = 2 * NN, ES = NB + 1, OS = MP | 1;
    extern __shared__ double sm[];
    double* su = sm;                        // [3][WX + 2][ES]
    double* so = sm + 3 * (WX + 2) * ES;    // [WX][OS]
    const int ntx = (a.nx + WX - 1) / WX, ex0 = int(blockIdx.x % ntx) * WX, ey = blockIdx.x / ntx;
    load_rows<NB, ES>(a, ex0, ey, su);
    __syncthreads();
    const int lane = threadIdx.x % 32, dir = (threadIdx.x / 32) / K, m = (threadIdx.x / 32) % K;
    const int ex = ex0 + lane;
    double r[K];
    if (ex < a.nx) {
        const int stride = dir == 0 ? 1 : N, at = dir * NN + (dir == 0 ? m * N : m);
        const double* u = su + ((WX + 2) + lane + 1) * ES + at;
        const int nb = dir == 0 ? ES : (WX + 2) * ES;
        double fe, fo;
        end_traces<N>(a, dir, ex, ey, u, stride, nb, -0.5, fe, fo);
        double se = 0.0, so_ = 0.0;   // sums of the even / odd entries above q
#pragma unroll
        for (int q = N - 1; q >= 0; --q) {
            if (q < K) r[q < K ? q : 0] = a.hl[dir][q] * (q % 2 == 0 ? fma(-2.0, so_, fe) : fma(-2.0, se, fo));
            double& b = q % 2 == 0 ? se : so_;
            b = fma(kRoot[q], u[q * stride], b);
        }
        if (dir == 0) {
#pragma unroll
            for (int q = 0; q < K; ++q) so[lane * OS + m * K + q] = r[q];
        }
    }
    __syncthreads();
    if (ex < a.nx && dir == 1) {
#pragma unroll
        for (int q = 0; q < K; ++q) so[lane * OS + q * K + m] += r[q];
    }
    __syncthreads();
    const int n = (min(ex0 + WX, a.nx) - ex0) * MP;
    double* g = a.out + (size_t(ey) * a.nx + ex0) * MP;
    for (int q = threadIdx.x; q < n; q += blockDim.x) g[q] = so[(q / MP) * OS + q % MP];
}

template <int N, bool TRANSPOSE>
void launch_div(const DivArgs& a, cudaStream_t s) {
    constexpr int K = N - 1, MP = K * K, NB = 2 * N * N;
    constexpr int IN = TRANSPOSE ? NB + 1 : (MP | 1), OUT = TRANSPOSE ? (MP | 1) : NB + 1;
    constexpr size_t smem = (size_t(3) * (WX + 2) * IN + size_t(WX) * OUT) * sizeof(double);
    static_assert(smem <= 227 * 1024, "three rows of elements fit shared memory");
    void (*const kernel)(DivArgs) = TRANSPOSE ? k_div_Bt<N> : k_div_B<N>;
    static const bool attr = [kernel] {   // once per process, thread-safe
        SIP_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
        return true;
    }();
    (void)attr;
    launch_k(kernel, dim3(unsigned(((a.nx + WX - 1) / WX) * a.ny)), WX * 2 * K, smem, s, a);
    SIP_CHECK_LAUNCH();
}

template <bool TRANSPOSE>
void launch_div_k(int k, const OpGeom& g, const double* in, double* out, cudaStream_t s) {
    DivArgs a{in, out, g.nx, g.ny, {g.bc[0], g.bc[1], g.bc[2], g.bc[3]}, {}};
    for (int q = 0; q <= k; ++q) {
        // the root with its rounding error, so that the products round once
        const double x = 2.0 * q + 1.0, l = std::sqrt(x), d = std::fma(-l, l, x) / (2.0 * l);
        for (int dir = 0; dir < 2; ++dir) {
            const double h = 0.25 * (dir == 0 ? g.hy : g.hx);
            a.hl[dir][q] = std::fma(h, l, h * d);
        }
    }
    switch (k + 1) {
        case 2: launch_div<2, TRANSPOSE>(a, s); break;
        case 3: launch_div<3, TRANSPOSE>(a, s); break;
        case 4: launch_div<4, TRANSPOSE>(a, s); break;
        case 5: launch_div<5, TRANSPOSE>(a, s); break;
        case 6: launch_div<6, TRANSPOSE>(a, s); break;
        case 7: launch_div<7, TRANSPOSE>(a, s); break;
        default: throw Error(SIP_ERR_INVALID_ARG, "unsupported polynomial degree");
    }
}

}  // namespace

template <>
void launch_apply_B<double>(int k, const OpGeom& g, const double* p, double* y, cudaStream_t s) {
    if (g.fp64) launch_apply_B_modes<double>(k, g, p, y, s);
    else launch_div_k<false>(k, g, p, y, s);
}
template <>
void launch_apply_Bt<double>(int k, const OpGeom& g, const double* u, double* y, cudaStream_t s) {
    if (g.fp64) launch_apply_Bt_modes<double>(k, g, u, y, s);
    else launch_div_k<true>(k, g, u, y, s);
}

}  // namespace sip
