// SIP apply with FP64-accurate results in 64-bit fixed point (fix_core.cuh):
// the FP64 operator for k <= 5 (but for Stokes solves of stiff problems: geom_solve in
// sip_solver.h), and the part of the FP32 operator that needs
// FP64 arithmetic (split precision: FP32 storage, the tiles of hi_tiles).
//
// What bounds it: instruction fetch and the latency of integer chains with the 12 to
// 16 warps per SM that shared memory admits (first stalls no_instruction and wait; the
// ALU pipe 50 % busy, the FP64 pipe 35 %, 47 % of the issue slots used at 512^2, k = 4).
// 17.6 thousand integer thread instructions per element at k = 3, 25.8 at k = 4.
// FP64 only converts, one multiply and one conversion per entry in (the halo's too:
// 1.5 times the tile's entries at 8 x 8, 1.75 at 8 x 4) and out: 171 operations per
// element at k = 3, 289 at k = 4, against the 933 of the FP64 kernel at k = 3, on a pipe
// that does 2 per SM and clock.  128^2, k = 3: 20.5 us, FP64 kernels 41.6; 512^2, k = 4:
// 459 and 736 us; 64^2, k = 3: 13.6 us.
//
// Layout: a CTA serves a tile of TW x TH elements with one thread per
// (element, line), both components; a warp shares its line index, lanes are
// elements.  The tile's and halo's entries are read once, a warp per element
// with consecutive lanes on consecutive entries, converted and kept in shared
// memory as integers; traces of all faces and the constant modes' jumps, once per
// face, go beside them, then rows and columns are two passes, and the results leave
// as consecutive stores.  (Jumps formed by each line that uses them cost 9 to 20 % more
// than once per face, and per element a CTA per SM at k = 4.)
#include "fix_core.cuh"
#include "sip_elem.cuh"
#include "sip_face.cuh"
#include "sip_internal.h"

namespace sip {

namespace {

// Entry (c, j, i) of A x on element (ex, ey) by the FP64 formulas, read from
// global memory: tiles with infinities, NaN or magnitudes outside the
// fixed-point range (E_MIN, E_MAX, ETA_E).  Zero table entries are skipped, so
// a NaN reaches the entries that depend on it and no others.
template <int N, typename TS>
__device__ __noinline__ double fp64_entry(const FixArgs<TS>& a, int ex, int ey, int q) {
    constexpr int NN = N * N, NB = 2 * NN;
    const int c = q / NN, j = (q / N) % N, i = q % N;
    const auto u = [&](size_t e, int cc, int jj, int ii) {
        return double(a.x[e * NB + cc * NN + jj * N + ii]);
    };
    const size_t e = size_t(ey) * a.nx + ex;
    const double etaK = double(a.eta[e]), hx = a.hx, hy = a.hy;
    const double sx = etaK * (c == 0 ? 2.0 : 1.0) * hy / hx;
    const double sy = etaK * (c == 0 ? 1.0 : 2.0) * hx / hy;
    double y = 0.0;
    for (int p = 0; p < N; ++p) {
        if (kT<N>.G[i][p] != 0.0) y += sx * kT<N>.G[i][p] * u(e, c, j, p);
        if (kT<N>.G[j][p] != 0.0) y += sy * kT<N>.G[j][p] * u(e, c, p, i);
        for (int r = 0; r < N; ++r) {
            const double dj = c == 0 ? kT<N>.D[r][j] : kT<N>.D[j][r];
            const double di = c == 0 ? kT<N>.D[i][p] : kT<N>.D[p][i];
            if (dj != 0.0 && di != 0.0) y += etaK * dj * di * u(e, 1 - c, r, p);
        }
    }
    double Dm[NN];
    for (int p = 0; p < NN; ++p) Dm[p] = kT<N>.D[p / N][p % N];
    for (int F = 0; F < 4; ++F) {
        const int dir = F / 2;
        const double sg = F & 1 ? 1.0 : -1.0;
        const fix::Mesh g{a.nx, a.ny, 0, 0, {a.bc[0], a.bc[1], a.bc[2], a.bc[3]}};
        const bool in = fix::has_nbr(g, ex, ey, F);
        const size_t en = F == 0 ? e - 1 : (F == 1 ? e + 1 : (F == 2 ? e - a.nx : e + a.nx));
        const double etaN = in ? double(a.eta[en]) : etaK;
        const double two_h = 2.0 / (dir == 0 ? hx : hy);
        double tr[2][4 * N];   // own, neighbour: [val c0 | val c1 | der c0 | der c1]
        for (int o = 0; o < 2; ++o) {
            const bool plus = ((F & 1) != 0) == (o == 0);
            for (int cc = 0; cc < 2; ++cc)
                for (int m = 0; m < N; ++m) {
                    double v = 0.0, d = 0.0;
                    for (int p = 0; p < N && (o == 0 || in); ++p) {
                        const double w = dir == 0 ? u(o ? en : e, cc, m, p) : u(o ? en : e, cc, p, m);
                        const double sv = plus || p % 2 == 0 ? 1.0 : -1.0;
                        const double sd = plus || p % 2 == 1 ? 1.0 : -1.0;
                        v += sv * kT<N>.lp[p] * w;
                        if (p > 0) d += sd * kT<N>.dp[p] * two_h * w;
                    }
                    tr[o][cc * N + m] = v;
                    tr[o][2 * N + cc * N + m] = d;
                }
        }
        const double pen = dir == 0 ? a.pen_x : a.pen_y;
        const double sigma = in ? pen * (etaK > etaN ? etaK : etaN) : 2.0 * pen * etaK;
        const FaceGeo<double> fg = dir == 0 ? make_face_geo<double>(hx, hy) : make_face_geo<double>(hy, hx);
        const int m = dir == 0 ? j : i, nq = dir == 0 ? i : j;
        double P, Q;
        face_pq<N, double>(in ? 0 : 1 + a.bc[F], c, m, dir, sg, fg, etaK, etaN, sigma, tr[0],
                           tr[0] + 2 * N, tr[1], tr[1] + 2 * N, Dm, P, Q);
        const double sv = F & 1 || nq % 2 == 0 ? 1.0 : -1.0;
        const double sd = F & 1 || nq % 2 == 1 ? 1.0 : -1.0;
        y += sv * kT<N>.lp[nq] * P;
        if (nq > 0) y += sd * kT<N>.dp[nq] * Q;
    }
    return y;
}

// Phase 0: entries and viscosities of the tile and its halo into shared
// memory as integers; returns whether this thread met a value outside the
// fixed-point range.
template <int N, int TW, int TH, typename TS>
__device__ __forceinline__ bool fix_load(const FixArgs<TS>& a, const fix::Mesh& g, fix::i64* sm) {
    using L = fix::Tile<N, TW, TH>;
    constexpr int SEG = N == 2 ? 8 : 32;              // lanes per element
    constexpr int EPW = 32 / SEG;                     // elements per warp
    constexpr int CH = (L::NB + SEG - 1) / SEG;       // entries per lane
    constexpr int U = CH == 1 ? 6 : (CH == 2 ? 3 : 2);   // elements in flight per lane group
    constexpr int STEP = L::NT / SEG;                 // lane groups of the CTA
    fix::i64* su = sm + L::O_U;
    double* seta = reinterpret_cast<double*>(sm + L::O_ETA);
    int* se = reinterpret_cast<int*>(sm + L::O_E);
    bool bad = false;
    for (int s = threadIdx.x; s < L::NS; s += L::NT) {
        int ex, ey;
        double v = 1.0;
        if (fix::staged_at<N, TW, TH>(g, s, ex, ey)) v = double(a.eta[size_t(ey) * a.nx + ex]);
        const long long b = fix::bits_of(v) >> 52;
        bad = bad || b < 1023 - fix::ETA_E || b > 1023 + fix::ETA_E;
        seta[s] = v;
    }
    const int grp = (threadIdx.x / 32) * EPW + (threadIdx.x % 32) / SEG, ls = threadIdx.x % SEG;
    // this lane's entries: conversion factor, component, whether it is a constant mode,
    // and the bits of its magnitude that count for either component's exponent
    double ss[CH];
    bool second[CH], mean[CH];
    unsigned of0[CH], of1[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        const int q = ls + c * SEG;
        ss[c] = a.ss[q % L::NN];
        second[c] = q >= L::NN;
        mean[c] = q == 0 || q == L::NN;
        of0[c] = mean[c] || second[c] ? 0u : 0x7fffffffu;
        of1[c] = mean[c] || !second[c] ? 0u : 0x7fffffffu;
    }
    // every lane of a warp takes the same number of rounds (shuffles below)
    constexpr int ROUNDS = (L::NS + STEP * U - 1) / (STEP * U);
#pragma unroll 1
    for (int r = 0; r < ROUNDS; ++r) {
        double v[U][CH];
        bool ok[U];
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const int s = (r * U + t) * STEP + grp;
            int ex, ey;
            ok[t] = s < L::NS && fix::staged_at<N, TW, TH>(g, s, ex, ey);
            const TS* p = a.x + (ok[t] ? (size_t(ey) * a.nx + ex) * L::NB : 0);
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int q = ls + c * SEG;
                v[t][c] = ok[t] && q < L::NB ? double(p[q]) : 0.0;
            }
        }
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const int s = (r * U + t) * STEP + grp;
            // largest magnitude (high words) of each component but its constant mode
            unsigned m0 = 0, m1 = 0;
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const unsigned h = unsigned(__double2hiint(v[t][c]));
                m0 = max(m0, h & of0[c]);
                m1 = max(m1, h & of1[c]);
            }
            if constexpr (SEG == 32) {
                m0 = __reduce_max_sync(0xffffffffu, m0);
                m1 = __reduce_max_sync(0xffffffffu, m1);
            } else {
#pragma unroll
                for (int o = SEG / 2; o > 0; o >>= 1) {
                    m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, o));
                    m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, o));
                }
            }
            const int e0 = int(m0 >> 20), e1 = int(m1 >> 20);
            int* above = reinterpret_cast<int*>(su + s * L::XS + L::NB);   // fix::mean_pack
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int q = ls + c * SEG;
                const unsigned h = unsigned(__double2hiint(v[t][c])) & 0x7fffffffu;
                const int ec = second[c] ? e1 : e0, e = mean[c] ? int(h >> 20) : ec;   // grid of this entry
                const bool fits = e >= fix::E_MIN && e <= fix::E_MAX;
                // outside the range, unless zero
                bad = bad || (!fits && (h | unsigned(__double2loint(v[t][c]))) != 0);
                if (s < L::NS && q < L::NB) {
                    su[s * L::XS + q] = fits ? fix::to_int(v[t][c] * fix::in_factor<N>(ss[c], e)) : 0;
                    if (mean[c]) above[second[c] ? 1 : 0] = e - ec;
                }
            }
            if (s < L::NS && ls == 0) se[s] = fix::expo_pack(e0, e1);
        }
    }
    return bad;
}

// y = alpha A x + beta z of the tile at (ex0, ey0), or with a.r1 the Q^2_1
// modes of that result.
template <int N, int TW, int TH, typename TS>
__device__ __forceinline__ void fix_body(const FixArgs<TS>& a, int ex0, int ey0) {
    using L = fix::Tile<N, TW, TH>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fix::i64* sm = reinterpret_cast<fix::i64*>(smem_raw);
    const fix::Mesh g{a.nx, a.ny, ex0, ey0, {a.bc[0], a.bc[1], a.bc[2], a.bc[3]}};
    const int tid = threadIdx.x;
    fix::i64* sw = sm + L::O_W;
    if (__syncthreads_or(fix_load<N, TW, TH, TS>(a, g, sm))) {
        for (int q = tid; q < L::NEL * L::NB; q += L::NT) {
            const int el = q / L::NB, m = q % L::NB;
            int ex, ey;
            if (fix::staged_at<N, TW, TH>(g, el, ex, ey))
                sw[m * L::EP + el] = fix::bits_of(a.alpha * fp64_entry<N, TS>(a, ex, ey, m));
        }
    } else {
        fix::phase_traces<N, TW, TH>(tid, g, sm);
        __syncthreads();
        fix::phase_lines<N, TW, TH, 0>(tid, g, a.k, a.os, sm);
        __syncthreads();
        fix::phase_lines<N, TW, TH, 1>(tid, g, a.k, a.os, sm);
    }
    __syncthreads();
    const double* sy = reinterpret_cast<const double*>(sw);
    if (a.r1) {
        for (int q = tid; q < L::NEL * 8; q += L::NT) {
            const int el = q / 8, l = q % 8, c = l / 4, j = (l / 2) % 2, i = l % 2;
            int ex, ey;
            if (!fix::staged_at<N, TW, TH>(g, el, ex, ey)) continue;
            const size_t e = size_t(ey) * a.nx + ex;
            const int m = c * L::NN + j * N + i;
            double w = sy[m * L::EP + el];
            if (a.z) w += a.beta * double(a.z[e * L::NB + m]);
            a.r1[e * 8 + l] = TS(w);
        }
        return;
    }
    // two entries of one element per thread (NB is even)
#pragma unroll 4
    for (int q = tid; q < L::NEL * L::NB / 2; q += L::NT) {
        const int el = q / (L::NB / 2), m = 2 * (q % (L::NB / 2));
        int ex, ey;
        if (!fix::staged_at<N, TW, TH>(g, el, ex, ey)) continue;
        const size_t o = (size_t(ey) * a.nx + ex) * L::NB + m;
        double w0 = sy[m * L::EP + el], w1 = sy[(m + 1) * L::EP + el];
        if (a.vec) {
            using V = typename std::conditional<sizeof(TS) == 8, double2, float2>::type;
            if (a.z) {
                const V zv = *reinterpret_cast<const V*>(a.z + o);
                w0 += a.beta * double(zv.x);
                w1 += a.beta * double(zv.y);
            }
            V out;
            out.x = TS(w0);
            out.y = TS(w1);
            *reinterpret_cast<V*>(a.y + o) = out;
        } else {
            if (a.z) {
                w0 += a.beta * double(a.z[o]);
                w1 += a.beta * double(a.z[o + 1]);
            }
            a.y[o] = TS(w0);
            a.y[o + 1] = TS(w1);
        }
    }
}

// CTAs per SM asked of the register allocator: what shared memory admits,
// with at least 96 registers a thread
template <int N, int TW, int TH>
constexpr int min_blocks() {
    using L = fix::Tile<N, TW, TH>;
    const int fit = int((228 * 1024) / (L::BYTES + 1024)), reg = 65536 / (L::NT * 96);
    const int b = fit < reg ? fit : reg;
    return b > 4 ? 4 : (b > 1 ? b : 1);   // more CTAs only serve meshes too small to fill them
}

template <int N, int TW, int TH, typename TS>
__global__ void __launch_bounds__(TW* TH* N, (min_blocks<N, TW, TH>())) k_apply_fix(const FixArgs<TS> a) {
    grid_dep_wait();
    const int ntx = (a.nx + TW - 1) / TW;   // 1D grid: no limit on mesh rows
    fix_body<N, TW, TH, TS>(a, int(blockIdx.x % ntx) * TW, int(blockIdx.x / ntx) * TH);
}

// Tiles of 32 x 2 elements named by a list (split precision), two CTAs each.
template <int N, typename TS>
__global__ void __launch_bounds__(32 * N, (min_blocks<N, 16, 2>())) k_apply_fix_list(const FixArgs<TS> a,
                                                                                 const int* __restrict__ tiles,
                                                                                 int ntx) {
    grid_dep_wait();
    const int t = tiles[blockIdx.x >> 1];
    const int ex0 = (t % ntx) * 32 + (blockIdx.x & 1) * 16;
    if (ex0 >= a.nx) return;
    fix_body<N, 16, 2, TS>(a, ex0, (t / ntx) * 2);
}

// Many operators in one launch, members with active[m] == 0 skipped.  SPLIT: CTAs
// 2b and 2b + 1 apply the operator of member items[b].x on its 32 x 2 tile
// items[b].y (split-precision tiles); else CTA b on its 8 x 4 tile.
template <int N, typename TS, bool SPLIT>
__global__ void __launch_bounds__(32 * N, (min_blocks<N, 16, 2>()))
    k_apply_fix_batch(const FixArgs<TS>* __restrict__ args, const int2* __restrict__ items,
                      const int* __restrict__ active) {
    grid_dep_wait();
    const int2 it = items[SPLIT ? blockIdx.x >> 1 : blockIdx.x];
    if (active && !active[it.x]) return;
    const FixArgs<TS>& a = args[it.x];
    if constexpr (SPLIT) {
        const int ntx = (a.nx + 31) / 32;
        const int ex0 = (it.y % ntx) * 32 + (blockIdx.x & 1) * 16;
        if (ex0 >= a.nx) return;
        fix_body<N, 16, 2, TS>(a, ex0, (it.y / ntx) * 2);
    } else {
        const int ntx = (a.nx + 7) / 8;
        fix_body<N, 8, 4, TS>(a, (it.y % ntx) * 8, (it.y / ntx) * 4);
    }
}

template <int N, int TW, int TH, typename TS>
void launch_tiles(const FixArgs<TS>& a, cudaStream_t s) {
    constexpr size_t smem = fix::Tile<N, TW, TH>::BYTES;
    static const bool attr = [] {   // once per process, thread-safe
        SIP_CUDA(cudaFuncSetAttribute(k_apply_fix<N, TW, TH, TS>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
        return true;
    }();
    (void)attr;
    launch_k(k_apply_fix<N, TW, TH, TS>, dim3(unsigned(((a.nx + TW - 1) / TW) * ((a.ny + TH - 1) / TH))),
             TW * TH * N, smem, s, a);
    SIP_CHECK_LAUNCH();
}

// Tile shape: large tiles convert fewer halo entries; meshes whose large tiles
// would leave SMs without a CTA take 8 x 4.
template <int N>
void launch_mesh(const FixArgs<double>& a, cudaStream_t s) {
    constexpr int TW = N == 2 ? 16 : 8, TH = N <= 4 ? 8 : 4;
    if (TH > 4 && (long long)((a.nx + TW - 1) / TW) * ((a.ny + TH - 1) / TH) < kSMs)
        launch_tiles<N, 8, 4, double>(a, s);
    else
        launch_tiles<N, TW, TH, double>(a, s);
}

template <int N>
void launch_list(const FixArgs<float>& a, const int* tiles, int n, cudaStream_t s) {
    constexpr size_t smem = fix::Tile<N, 16, 2>::BYTES;
    static const bool attr = [] {
        SIP_CUDA(cudaFuncSetAttribute(k_apply_fix_list<N, float>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
        return true;
    }();
    (void)attr;
    launch_k(k_apply_fix_list<N, float>, dim3(unsigned(2 * n)), 32 * N, smem, s, a, tiles,
             (a.nx + 31) / 32);
    SIP_CHECK_LAUNCH();
}

template <int N, typename TS, bool SPLIT>
void launch_batch(const FixArgs<TS>* args, const int2* items, int n, const int* active, cudaStream_t s) {
    constexpr size_t smem = SPLIT ? fix::Tile<N, 16, 2>::BYTES : fix::Tile<N, 8, 4>::BYTES;
    static const bool attr = [] {
        SIP_CUDA(cudaFuncSetAttribute(k_apply_fix_batch<N, TS, SPLIT>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
        return true;
    }();
    (void)attr;
    launch_k(k_apply_fix_batch<N, TS, SPLIT>, dim3(unsigned(SPLIT ? 2 * n : n)), 32 * N, smem, s, args,
             items, active);
    SIP_CHECK_LAUNCH();
}

}  // namespace

template <typename TS>
bool make_fix_args(int N, const OpGeom& g, const TS* x, TS* y, const TS* eta, double alpha, const TS* z,
                   double beta, TS* r1, FixArgs<TS>& a) {
    if (N < 2 || N > 6 || !(std::fabs(alpha) > 1e-9 && std::fabs(alpha) < 1e9)) return false;
    const double r = g.hy / g.hx, ch = 0.5 * g.pen_x * g.hx;
    if (!(std::fabs(0.5 * g.pen_y * g.hy - ch) <= 1e-12 * std::fabs(ch))) return false;
    switch (N) {
        case 2: a.k = fix::make_scal<2>(r, ch); break;
        case 3: a.k = fix::make_scal<3>(r, ch); break;
        case 4: a.k = fix::make_scal<4>(r, ch); break;
        case 5: a.k = fix::make_scal<5>(r, ch); break;
        default: a.k = fix::make_scal<6>(r, ch); break;
    }
    if (!a.k.ok) return false;
    a.x = x;
    a.y = y;
    a.eta = eta;
    a.z = z;
    a.r1 = r1;
    a.alpha = alpha;
    a.beta = beta;
    a.nx = g.nx;
    a.ny = g.ny;
    a.hx = g.hx;
    a.hy = g.hy;
    a.pen_x = g.pen_x;
    a.pen_y = g.pen_y;
    for (int i = 0; i < 4; ++i) a.bc[i] = g.bc[i];
    const uintptr_t two = 2 * sizeof(TS) - 1;
    a.vec = (reinterpret_cast<uintptr_t>(y) & two) == 0 && (reinterpret_cast<uintptr_t>(z) & two) == 0;
    for (int j = 0; j < N; ++j)
        for (int i = 0; i < N; ++i) {
            a.ss[j * N + i] = std::sqrt((2.0 * i + 1.0) * (2.0 * j + 1.0)) / 2.0;
            a.os[j * N + i] = alpha * a.ss[j * N + i];
        }
    return true;
}
template bool make_fix_args<double>(int, const OpGeom&, const double*, double*, const double*, double,
                                    const double*, double, double*, FixArgs<double>&);
template bool make_fix_args<float>(int, const OpGeom&, const float*, float*, const float*, double,
                                   const float*, double, float*, FixArgs<float>&);

bool launch_apply_fix(int N, const OpGeom& g, const double* x, double* y, const double* eta,
                      double alpha, const double* z, double beta, double* r1, cudaStream_t s) {
    FixArgs<double> a;
    if (!make_fix_args<double>(N, g, x, y, eta, alpha, z, beta, r1, a)) return false;
    switch (N) {
        case 2: launch_mesh<2>(a, s); return true;
        case 3: launch_mesh<3>(a, s); return true;
        case 4: launch_mesh<4>(a, s); return true;
        case 5: launch_mesh<5>(a, s); return true;
        default: launch_mesh<6>(a, s); return true;
    }
}

bool launch_apply_fix_list(int N, const OpGeom& g, const float* x, float* y, const float* eta,
                           float alpha, const float* z, float beta, float* r1, cudaStream_t s) {
    FixArgs<float> a;
    if (!make_fix_args<float>(N, g, x, y, eta, alpha, z, beta, r1, a)) return false;
    switch (N) {
        case 2: launch_list<2>(a, g.hi_tiles, g.n_hi, s); return true;
        case 3: launch_list<3>(a, g.hi_tiles, g.n_hi, s); return true;
        case 4: launch_list<4>(a, g.hi_tiles, g.n_hi, s); return true;
        case 5: launch_list<5>(a, g.hi_tiles, g.n_hi, s); return true;
        default: launch_list<6>(a, g.hi_tiles, g.n_hi, s); return true;
    }
}

int fix_tile_count(int nx, int ny) { return ((nx + 7) / 8) * ((ny + 3) / 4); }

template <typename TS>
void launch_apply_fix_batch(int N, const FixArgs<TS>* args, const int2* items, int n_items,
                            const int* active, cudaStream_t s) {
    if (n_items <= 0) return;
    constexpr bool SPLIT = sizeof(TS) == 4;
    switch (N) {
        case 2: launch_batch<2, TS, SPLIT>(args, items, n_items, active, s); break;
        case 3: launch_batch<3, TS, SPLIT>(args, items, n_items, active, s); break;
        case 4: launch_batch<4, TS, SPLIT>(args, items, n_items, active, s); break;
        case 5: launch_batch<5, TS, SPLIT>(args, items, n_items, active, s); break;
        case 6: launch_batch<6, TS, SPLIT>(args, items, n_items, active, s); break;
        default: throw Error(SIP_ERR_INVALID_ARG, "batched apply: degree above 5");
    }
}
template void launch_apply_fix_batch<double>(int, const FixArgs<double>*, const int2*, int, const int*,
                                             cudaStream_t);
template void launch_apply_fix_batch<float>(int, const FixArgs<float>*, const int2*, int, const int*,
                                            cudaStream_t);

}  // namespace sip
