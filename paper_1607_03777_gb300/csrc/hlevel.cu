// One continuous level of the h-hierarchy in two launches: everything before
// the coarse correction (Chebyshev / point-Jacobi steps from zero, residual,
// restriction) and everything after it (interpolation, steps).
//
// What bounds it: launches and latency.  A stencil application on a 129^2-vertex level is
// 1 us of FP64 work and 4 MB from L2, but one launch per step takes about 4 us
// in a replayed graph, nine per level.  Here a CTA runs all steps of its tile on
// a halo that shrinks by one ring per application, one thread per (vertex,
// component) with its stencil row in registers (read once instead of once per
// step) and the direction in shared memory.  The rings are recomputed by the
// neighbouring tiles: with three steps 1.6 (before) and 1.4 (after) stencil rows per row
// kept at 12 x 12 vertices, 3.2 and 2.4 at 4 x 4; FP64 levels where that work
// outweighs the launches keep one launch per step (fused_level_ok).  On 129^2 vertices
// the FP64 pipe is 76 % busy.
#include "sip_internal.h"
#include "sip_level.cuh"
#include "sip_solver.h"

namespace sip {

namespace {

constexpr int kMaxThreads = 768;
template <typename T>
__device__ __forceinline__ T row_dot(const T (&s)[18], const T* v, int rw) {
    T acc = T(0);
#pragma unroll
    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
            const T* w = v + 2 * ((dy - 1) * rw + dx - 1);
            const int t = 2 * (dy * 3 + dx);
            acc += s[t] * w[0] + s[t + 1] * w[1];
        }
    return acc;
}

template <typename T>
__device__ __forceinline__ void load_row(const T* S, size_t g, T (&s)[18]) {
    const T* p = S + (g / 2) * 36 + (g % 2) * 2;
#pragma unroll
    for (int t = 0; t < 9; ++t) ld2<T, true>(p + 4 * t, s[2 * t], s[2 * t + 1]);
}

// One thread's place in its tile's region.
struct Place {
    bool in;       // inside the grid
    int ring;      // distance from the region's edge
    int node;      // 2 * (local vertex) + component
    size_t g;      // global row
    int gx, gy, c;
};

template <typename T>
__device__ __forceinline__ Place place(const LevelArgs<T>& a, int ox, int oy) {
    Place p;
    p.c = threadIdx.x % 2;
    const int v = threadIdx.x / 2, lx = v % a.rw, ly = v / a.rw;
    p.node = threadIdx.x;
    p.gx = ox + lx;
    p.gy = oy + ly;
    p.in = ly < a.rw && p.gx >= 0 && p.gx < a.nvx && p.gy >= 0 && p.gy < a.nvy;
    p.ring = min(min(lx, a.rw - 1 - lx), min(ly, a.rw - 1 - ly));
    p.g = p.in ? 2 * (size_t(p.gy) * a.nvx + p.gx) + p.c : 0;
    return p;
}

// x = Chebyshev steps on S x = b from zero; bc = R_h (b - S x).
template <typename T>
__device__ __forceinline__ void level_before(const LevelArgs<T>& a, int tile) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nt = 2 * a.rw * a.rw;
    T* sd = reinterpret_cast<T*>(smem_raw);   // direction, then iterate
    T* sr = sd + nt;                          // residual
    const int ntx = (a.ncx + a.tile) / a.tile;   // ceil((ncx + 1) / tile)
    const int I0 = (tile % ntx) * a.tile, J0 = (tile / ntx) * a.tile;
    const Place p = place(a, 2 * I0 - 1 - a.steps, 2 * J0 - 1 - a.steps);
    const bool mine = int(threadIdx.x) < nt;
    T s[18], r = T(0), d = T(0), x = T(0), bv = T(0), di = T(0);
    if (p.in) {
        bv = a.b[p.g];
        di = a.dinv[p.g];
        if (p.ring > 0) load_row(a.S, p.g, s);
        r = bv;
        x = d = a.c2[0] * di * bv;
    }
    if (mine) sd[p.node] = d;
    __syncthreads();
    for (int st = 1; st < a.steps; ++st) {
        if (p.in && p.ring >= st) {
            r -= row_dot(s, sd + p.node - p.c, a.rw);
            d = a.c1[st] * d + a.c2[st] * di * r;
            x += d;
        }
        __syncthreads();
        if (mine) sd[p.node] = st + 1 < a.steps ? d : x;
        __syncthreads();
    }
    if (mine) sr[p.node] = p.in && p.ring >= a.steps ? bv - row_dot(s, sd + p.node - p.c, a.rw) : T(0);
    const int fx = p.gx - 2 * I0, fy = p.gy - 2 * J0, tf = 2 * a.tile;
    if (p.in && fx >= 0 && fx < tf && fy >= 0 && fy < tf) a.x[p.g] = x;
    __syncthreads();
    for (int q = threadIdx.x; q < 2 * a.tile * a.tile; q += blockDim.x) {
        const int c = q % 2, v = q / 2, I = I0 + v % a.tile, J = J0 + v / a.tile;
        if (I > a.ncx || J > a.ncy) continue;
        // the vertex in the region: 2 (I - I0) + 1 + steps
        const T* w = sr + 2 * ((2 * (J - J0) + 1 + a.steps) * a.rw + 2 * (I - I0) + 1 + a.steps) + c;
        T acc = T(0);
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                const T wt = (dy == 0 ? T(1) : T(0.5)) * (dx == 0 ? T(1) : T(0.5));
                acc += wt * w[2 * (dy * a.rw + dx)];   // zero outside the grid
            }
        a.bc[2 * (size_t(J) * (a.ncx + 1) + I) + c] = acc;
    }
}

// x = Chebyshev steps on S x = b from xin + P_h xc.
template <typename T>
__device__ __forceinline__ void level_after(const LevelArgs<T>& a, int tile) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nt = 2 * a.rw * a.rw;
    T* sd = reinterpret_cast<T*>(smem_raw);
    const int tf = 2 * a.tile, ntx = (a.nvx + tf - 1) / tf;
    const int X0 = (tile % ntx) * tf, Y0 = (tile / ntx) * tf;
    const Place p = place(a, X0 - a.steps, Y0 - a.steps);
    const bool mine = int(threadIdx.x) < nt;
    T s[18], r = T(0), d = T(0), x = T(0), bv = T(0), di = T(0);
    if (p.in) {
        bv = a.b[p.g];
        di = a.dinv[p.g];
        if (p.ring > 0) load_row(a.S, p.g, s);
        const T* q = a.xc + 2 * (size_t(p.gy / 2) * (a.ncx + 1) + p.gx / 2) + p.c;
        const int ux = p.gx % 2 ? 2 : 0, uy = p.gy % 2 ? 2 * (a.ncx + 1) : 0;
        T v = q[0];
        if (ux && uy) v = T(0.25) * (q[0] + q[ux] + q[uy] + q[ux + uy]);
        else if (ux || uy) v = T(0.5) * (q[0] + q[ux + uy]);
        x = a.xin[p.g] + v;
    }
    if (mine) sd[p.node] = x;
    __syncthreads();
    if (p.in && p.ring >= 1) {
        r = bv - row_dot(s, sd + p.node - p.c, a.rw);
        d = a.c2[0] * di * r;
    }
    T pend = d;
    for (int st = 1; st < a.steps; ++st) {
        __syncthreads();
        if (mine) sd[p.node] = d;
        __syncthreads();
        if (p.in && p.ring >= st + 1) {
            r -= row_dot(s, sd + p.node - p.c, a.rw);
            d = a.c1[st] * d + a.c2[st] * di * r;
            x += pend + d;
            pend = T(0);
        }
    }
    if (a.steps == 1) x += d;
    const int fx = p.gx - X0, fy = p.gy - Y0;
    if (p.in && fx >= 0 && fx < tf && fy >= 0 && fy < tf) a.x[p.g] = x;
}

template <typename T, bool AFTER>
__global__ void __launch_bounds__(kMaxThreads) k_level(const LevelArgs<T> a) {
    grid_dep_wait();
    if constexpr (AFTER) level_after<T>(a, blockIdx.x);
    else level_before<T>(a, blockIdx.x);
}

template <typename T, bool AFTER>
__global__ void __launch_bounds__(kMaxThreads) k_level_batch(const LevelArgs<T>* __restrict__ args,
                                                             const int2* __restrict__ items,
                                                             const int* __restrict__ active) {
    grid_dep_wait();
    const int2 it = items[blockIdx.x];
    if (active && !active[it.x]) return;
    const LevelArgs<T> a = args[it.x];
    if constexpr (AFTER) level_after<T>(a, it.y);
    else level_before<T>(a, it.y);
}

// Coarse vertices per tile and direction: the largest (least recomputation)
// that still gives most SMs (110 of 152) a tile.
int level_tile(int nvxc, int nvyc, int steps, int members) {
    for (int t = 6; t > 2; --t) {
        const int rw = 2 * t + 1 + 2 * steps;
        if (2 * rw * rw > kMaxThreads) continue;
        if (((nvxc + t - 1) / t) * ((nvyc + t - 1) / t) * members >= 110) return t;
    }
    return 2;
}

template <typename T>
LevelArgs<T> level_args(const HLevel<T>& L, const HLevel<T>& C, int steps, const double* c1,
                        const double* c2, T* x, int members) {
    LevelArgs<T> a{};
    a.nvx = L.nvx;
    a.nvy = L.nvy;
    a.ncx = C.nx;
    a.ncy = C.ny;
    a.S = L.S.template as<T>();
    a.dinv = L.dinv.template as<T>();
    a.b = L.b.template as<T>();
    a.x = x;
    a.steps = steps;
    a.tile = level_tile(C.nvx, C.nvy, steps, members);
    for (int i = 0; i < steps; ++i) {
        a.c1[i] = T(c1[i]);
        a.c2[i] = T(c2[i]);
    }
    return a;
}

inline int round32(int n) { return (n + 31) / 32 * 32; }

}  // namespace

// FP64: the recomputed rings cost more than the launches they save from about 130^2
// vertices on, over all members of a batch.  V-cycle, k = 1, two launches per level / one
// per step: 128^2 elements 164 / 179 us, 144^2 222 / 211, 192^2 268 / 232, 256^2 429 / 384;
// grouped batches, k = 2: 4 x 64^2 48.1 / 50.7 ms, 16 x 32^2 62.9 / 61.8, 8 x 64^2 86.7 / 83.3,
// 8 x 128^2 259 / 239.  FP32: 256^2 126 / 152 us, 512^2 352 / 351.
template <typename T>
bool fused_level_ok(int steps, size_t vertices) {
    if (steps < 1 || steps > kLevelSteps) return false;
    return sizeof(T) == 4 || vertices <= 17000;
}

template <typename T>
LevelArgs<T> level_before_args(HLevel<T>& L, HLevel<T>& C, int steps, const double* c1, const double* c2,
                               T* x, int members) {
    LevelArgs<T> a = level_args(L, C, steps, c1, c2, x, members);
    a.rw = 2 * a.tile + 1 + 2 * steps;
    a.bc = C.b.template as<T>();
    a.tiles = ((C.nvx + a.tile - 1) / a.tile) * ((C.nvy + a.tile - 1) / a.tile);
    a.threads = round32(2 * a.rw * a.rw);
    return a;
}

template <typename T>
LevelArgs<T> level_after_args(HLevel<T>& L, HLevel<T>& C, int steps, const double* c1, const double* c2,
                              const T* xin, T* x, int members) {
    LevelArgs<T> a = level_args(L, C, steps, c1, c2, x, members);
    const int tf = 2 * a.tile;
    a.rw = tf + 2 * steps;
    a.xin = xin;
    a.xc = C.x.template as<T>();
    a.tiles = ((L.nvx + tf - 1) / tf) * ((L.nvy + tf - 1) / tf);
    a.threads = round32(2 * a.rw * a.rw);
    return a;
}

template <typename T>
void launch_level(const LevelArgs<T>& a, cudaStream_t s) {
    const size_t smem = size_t(2) * a.threads * sizeof(T);   // two vectors of a tile's region
    if (a.xin)
        launch_k(k_level<T, true>, unsigned(a.tiles), unsigned(a.threads), smem, s, a);
    else
        launch_k(k_level<T, false>, unsigned(a.tiles), unsigned(a.threads), smem, s, a);
    SIP_CHECK_LAUNCH();
}

template <typename T>
void launch_level_batch(bool after, const LevelArgs<T>* args, const int2* items, int n_items, int threads,
                        const int* active, cudaStream_t s) {
    if (n_items <= 0) return;
    const size_t smem = size_t(2) * threads * sizeof(T);
    if (after)
        launch_k(k_level_batch<T, true>, unsigned(n_items), unsigned(threads), smem, s, args, items, active);
    else
        launch_k(k_level_batch<T, false>, unsigned(n_items), unsigned(threads), smem, s, args, items, active);
    SIP_CHECK_LAUNCH();
}

#define SIP_LEVEL(T)                                                                              \
    template bool fused_level_ok<T>(int, size_t);                                                 \
    template LevelArgs<T> level_before_args<T>(HLevel<T>&, HLevel<T>&, int, const double*,        \
                                               const double*, T*, int);                           \
    template LevelArgs<T> level_after_args<T>(HLevel<T>&, HLevel<T>&, int, const double*,         \
                                              const double*, const T*, T*, int);                  \
    template void launch_level<T>(const LevelArgs<T>&, cudaStream_t);                             \
    template void launch_level_batch<T>(bool, const LevelArgs<T>*, const int2*, int, int, const int*, \
                                        cudaStream_t);
SIP_LEVEL(double)
SIP_LEVEL(float)
#undef SIP_LEVEL

}  // namespace sip
