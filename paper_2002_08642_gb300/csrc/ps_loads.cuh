// ps_loads.cuh -- pressure loads on the mass points of the wing (Sec. 4.1,
// fluid-to-solid coupling paragraph): the static pressure interpolated to
// every node with a smoothed discrete delta function, and per triangle the
// force -p_v (A/3) n on each of its vertices.
//
// Kernel (the paper cites a smoothing technique for discrete delta functions
// without printing one; reading): the 4-point cosine kernel
// phi(r) = (1/4)(1 + cos(pi r/2)), |r| <= 2, convolved with the unit box,
//   phi_s(r) = (1/4)(1 + (2/pi)(sin(pi(r+1/2)/2) - sin(pi(r-1/2)/2))), |r| <= 3/2,
//   phi_s(r) = (1/4)((5/2 - |r|) - (2/pi) sin(pi(|r|-1/2)/2)),        3/2 < |r| < 5/2,
// zero beyond; five grid points per axis, periodic grid. All sums in double.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "ps_async.cuh"

namespace ps {

struct LoadArgs {
    int n, nz;            // grid n x n x nz, spacing dx on every axis
    double dx;
    const double* xw;     // n_nodes x 3, wing frame
    int n_nodes;
    const int32_t* tri;   // n_tri x 3
    int n_tri;
    double R[9], XO[3];   // wing frame -> global
};

// phi_s with one cosine: sin(pi(r+1/2)/2) - sin(pi(r-1/2)/2) = sqrt(2) cos(pi r/2)
// and sin(pi(r-1/2)/2) = cos(pi(r-3/2)/2), the arguments in units of pi.
__device__ __forceinline__ double delta_smoothed(double r) {
    r = fabs(r);
    if (!(r < 2.5)) return 0.0;   // also a node that is no number
    const bool inner = r <= 1.5;
    const double t = cospi(0.5 * (inner ? r : r - 1.5));
    return inner ? 0.25 * (1.0 + (2.0 * M_SQRT2 / M_PI) * t) : 0.25 * ((2.5 - r) - (2.0 / M_PI) * t);
}

// One warp per node v: p at the node from the 6 x 6 x 6 grid points around
// it, then F_v = -p_v sum over the triangles containing v of
// ((b - a) x (c - a)) / 6 (global frame).
//   weights   lane 6 r + q holds the delta weight of point q on axis r;
//   pressure  lane l sums the grid points l, l + 32, ... of the 216, then a
//             fixed shuffle tree;
//   triangles the lanes scan the list 32 at a time; the triangles that hold
//             v go to a list of 32 per warp in index order, and a full list
//             (and the rest) is summed with one triangle per lane.
// Everything is a fixed order: deterministic. FP64 issue bound (a warp's FP64
// instruction takes 64 cycles of a quarter SM), so the 18 weights and the
// triangles' cross products go side by side in the lanes instead of one after
// another: 833 nodes, 1600 triangles at 192^3, 19 us on a GB300 against 65 + 27 us with
// one thread per node (36 sines each) and a cross product per divergent match.
static constexpr int kLoadWarps = 4;
template <typename T>
__global__ void __launch_bounds__(32 * kLoadWarps)
k_node_loads(LoadArgs a, const T* __restrict__ pf, double* __restrict__ pn, double* __restrict__ F) {
    pdl_wait();
    __shared__ int hit[kLoadWarps][32];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int v = blockIdx.x * kLoadWarps + wid;
    if (v >= a.n_nodes) return;   // whole warps leave together
    const unsigned all = 0xffffffffu;
    // grid position of the node: lanes 0..2 one axis each
    double g = 0.0;
    if (lane < 3) {
        const double* x = a.xw + 3 * (size_t)v;
        const double* R = a.R + 3 * lane;
        g = (a.XO[lane] + R[0] * x[0] + R[1] * x[1] + R[2] * x[2]) / a.dx;
    }
    const int ax = lane < 18 ? lane / 6 : 0, q = lane % 6;
    g = __shfl_sync(all, g, ax);
    const double lo = floor(g) - 2.0;
    const double w = delta_smoothed(g - (lo + (double)q));
    // periodic grid index of this lane's point on its axis
    const long dim = ax == 2 ? a.nz : a.n;
    const int at = (int)((((long)lo + q) % dim + dim) % dim);
    double acc = 0.0;
#pragma unroll
    for (int m0 = 0; m0 < 216; m0 += 32) {
        const int m = m0 + lane, i = m / 36 % 6, j = m / 6 % 6, k = m % 6;   // m >= 216 only shuffles
        const double wx = __shfl_sync(all, w, i), wy = __shfl_sync(all, w, 6 + j), wz = __shfl_sync(all, w, 12 + k);
        const int xi = __shfl_sync(all, at, i), yj = __shfl_sync(all, at, 6 + j), zk = __shfl_sync(all, at, 12 + k);
        if (m < 216) acc += wx * wy * (wz * (double)pf[((size_t)xi * a.n + yj) * a.nz + zk]);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(all, acc, o);
    if (lane == 0) pn[v] = acc;

    double s[3] = {0.0, 0.0, 0.0};
    auto area = [&](int t) {   // s += (R (b - a)) x (R (c - a))
        const double* A = a.xw + 3 * (size_t)a.tri[3 * t];
        const double* B = a.xw + 3 * (size_t)a.tri[3 * t + 1];
        const double* C = a.xw + 3 * (size_t)a.tri[3 * t + 2];
        double d1[3], d2[3], e1[3], e2[3];
        for (int r = 0; r < 3; ++r) { d1[r] = B[r] - A[r]; d2[r] = C[r] - A[r]; }
        for (int r = 0; r < 3; ++r) {
            e1[r] = a.R[3 * r] * d1[0] + a.R[3 * r + 1] * d1[1] + a.R[3 * r + 2] * d1[2];
            e2[r] = a.R[3 * r] * d2[0] + a.R[3 * r + 1] * d2[1] + a.R[3 * r + 2] * d2[2];
        }
        s[0] += e1[1] * e2[2] - e1[2] * e2[1];
        s[1] += e1[2] * e2[0] - e1[0] * e2[2];
        s[2] += e1[0] * e2[1] - e1[1] * e2[0];
    };
    int n_hit = 0;
    constexpr int U = 4;   // groups of 32 triangles whose indices are in flight together
    for (int t0 = 0; t0 < a.n_tri; t0 += 32 * U) {
        int id[U][3];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int t = t0 + 32 * k + lane;
#pragma unroll
            for (int c = 0; c < 3; ++c) id[k][c] = t < a.n_tri ? a.tri[3 * t + c] : -1;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const bool in = (id[k][0] == v) | (id[k][1] == v) | (id[k][2] == v);
            const unsigned m = __ballot_sync(all, in);
            if (m == 0) continue;
            const int n_new = __popc(m);
            if (n_hit + n_new > 32) {   // the list is full: sum it
                if (lane < n_hit) area(hit[wid][lane]);
                __syncwarp();
                n_hit = 0;
            }
            if (in) hit[wid][n_hit + __popc(m & ((1u << lane) - 1u))] = t0 + 32 * k + lane;
            __syncwarp();
            n_hit += n_new;
        }
    }
    if (lane < n_hit) area(hit[wid][lane]);
    for (int o = 16; o > 0; o >>= 1)
        for (int r = 0; r < 3; ++r) s[r] += __shfl_down_sync(all, s[r], o);
    if (lane == 0) {
        const double f = -acc / 6.0;
        for (int r = 0; r < 3; ++r) F[3 * (size_t)v + r] = f * s[r];
    }
}

}  // namespace ps
