// ps_mask.cuh -- GPU rasteriser of the wing mask chi and the solid velocity
// u_s from the mass-spring wing's triangle mesh (Sec. 4.1):
//   * delta(x) = min over triangles of the distance from grid point x to the
//     triangle, each triangle tested only against the grid points of its
//     bounding box dilated by t_w + h (the mask's reach; no periodic images);
//   * chi(delta) by Eq. (mask_function) (or the tanh profile, evaluated at
//     every point against every triangle);
//   * u_s = V_O + R (sum_v beta_v v_v^(w)) + Omega x (x - X_O) with beta the
//     barycentric coordinates of the closest point on the closest triangle
//     (Eq. relative_velocities).
//
// Banded (cosine) profile, three kernels per call (five in FP64):
//   prepare   zero chi/u_s and reset the per-point keys of the points the
//             previous call touched (list kept in the workspace), clear the
//             line flags; the global node positions X_O + R x^(w) and
//             velocities R v^(w) (double); per triangle the grid-index bounding box and the geometry the
//             pair tests need, in the context precision;
//   pairs     a warp per triangle (several where there are few) walks the
//             points of its box. FP32: for every pair with distance < reach
//             an atomicMin of a 64-bit key, the squared distance's bits
//             (non-negative IEEE values order like their bit patterns) above
//             the triangle index, so that the minimum also names the winner
//             (exact ties -> smallest index); the first writer appends the
//             point to the touched list. FP64, three walks:
//               bound   an upper bound of each point's least squared
//                       distance, and the touched list, in FP32;
//               least   its exact value (atomicMin of the bits);
//               ties    pairs within a few ulps of it: atomicMin of the
//                       triangle index (near-ties -> smallest index);
//   evaluate  per touched point: distance and barycentrics recomputed in
//             double on the winning triangle, chi, u_s, line flags.
// The distance used to pick the winner is computed in the context precision.
//
// What bounds it: launches and FP64 issue (a warp's FP64 instruction takes 64
// cycles of a quarter SM whatever its lanes do). So the triangles' boxes go
// with the clearing instead of into a kernel of their own, one axis per lane;
// a warp owns a triangle, so that no prefix sum over the boxes and no search
// in it is needed; distances are compared squared (no root), the dot products
// of the edges are made once per triangle, divisions by constants are
// products; and the FP64 pair tests run only for the pairs that a FP32 lower
// bound of the distance leaves, 32 at a time.
// GB300, each kernel alone on the device, against clear + boxes + prefix sum +
// pair pass(es) + evaluate: 121 nodes at 48^3 FP32 48 -> 28 us (6 + 5 + 17),
// 600 nodes at 128^3 FP64 229 -> 107 us (8 + 24 + 29 + 29 + 17). Then sign tests
// and bound conversions on the integer pipe, the cosine as a series on its half
// period and node velocities rotated once: wing 48^3 663 -> 632 us (8 steps),
// 128^3 FP64 3000 -> 2896 (2 steps), FP64 gradient window 64^3 8.9 -> 8.4 ms.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "ps_async.cuh"

#include <string>

namespace ps {

struct MaskArgs {
    int n, nz;   // grid n x n x nz, spacing dx on every axis
    int x_lo, x_hi;   // x-planes [x_lo, x_hi) rasterised (a slab of the sharded step; 0, n otherwise)
    double dx, inv_dx, tw, h;
    int profile;
    const double* xw;
    const double* vw;
    int n_nodes;
    const int32_t* tri;
    int n_tri;
    double R[9], XO[3], VO[3], Om[3];
};

static constexpr int kMaskMaxTri = 1 << 17;
static constexpr int kMaskMaxNodes = 1 << 17;

// Per-triangle geometry of the pair tests: bounding box dilated by the reach
// (first grid index and extent per axis); vertex a = ca dx + f per axis (ca
// its grid cell index, f the rest, about [0, dx)), edges b - a and c - a and
// their dot products; the lengths rounded once from double to T. A grid point
// minus a is then (i - ca) dx - f, with no double arithmetic per pair.
// m, r: a sphere around the triangle (centre relative to a); nrm: the unit
// normal, 0 for a triangle without a plane (has_plane; such a one gives no bounds).
template <typename T> struct TriGeo {
    int i0[3], e[3], ca[3];
    float r;
    T f[3], b[3], c[3];
    T bb, bc, cc;
    float m[3], nrm[3];
};
static constexpr size_t kTriGeoBytes = 160;   // >= sizeof(TriGeo<double>)
static_assert(sizeof(TriGeo<double>) <= kTriGeoBytes, "triangle geometry slot");

// Workspace: keys (8 B/pt), winner ids (4 B/pt), two touched lists (4 B/pt
// each), counters, node and triangle scratch.
inline size_t mask_workspace_bytes(int n, int nz) {
    const size_t n3 = (size_t)n * n * nz;
    auto a = [](size_t x) { return (x + 255) & ~(size_t)255; };
    return a(n3 * 8) + a(n3 * 4) + 2 * a(n3 * 4) + a(64) + 2 * a((size_t)kMaskMaxNodes * 3 * 8) +
           a((size_t)kMaskMaxTri * kTriGeoBytes);
}

struct MaskWs {
    unsigned long long* key;
    int32_t* win;
    uint32_t* list[2];
    unsigned long long* cnt;  // [0],[1]: list lengths, [4]: bad-index flag
    double* xg;                // node positions, global
    double* vg;                // R times the wing-frame node velocities
    unsigned char* geo;        // per triangle: TriGeo<T> in kTriGeoBytes
};

inline MaskWs mask_ws_split(unsigned char* w, int n, int nz) {
    const size_t n3 = (size_t)n * n * nz;
    auto a = [](size_t x) { return (x + 255) & ~(size_t)255; };
    MaskWs m;
    size_t o = 0;
    m.key = (unsigned long long*)(w + o); o += a(n3 * 8);
    m.win = (int32_t*)(w + o); o += a(n3 * 4);
    m.list[0] = (uint32_t*)(w + o); o += a(n3 * 4);
    m.list[1] = (uint32_t*)(w + o); o += a(n3 * 4);
    m.cnt = (unsigned long long*)(w + o); o += a(64);
    m.xg = (double*)(w + o); o += a((size_t)kMaskMaxNodes * 3 * 8);
    m.vg = (double*)(w + o); o += a((size_t)kMaskMaxNodes * 3 * 8);
    m.geo = w + o;
    return m;
}

// Closest point of triangle (a, b, c) to p by Voronoi-region tests on the
// vertices, edges and face (the published closest-point-on-triangle method
// of Ericson, Real-Time Collision Detection, Sec. 5.1.5); returns squared
// distance and barycentrics.
template <typename R>
__device__ __forceinline__ R closest_tri(const R p[3], const R a[3], const R b[3], const R c[3], R bary[3]) {
    R ab[3], ac[3], ap[3], bp[3], cp[3];
    for (int i = 0; i < 3; ++i) {
        ab[i] = b[i] - a[i];
        ac[i] = c[i] - a[i];
        ap[i] = p[i] - a[i];
        bp[i] = p[i] - b[i];
        cp[i] = p[i] - c[i];
    }
    auto dot = [](const R* u, const R* v) { return u[0] * v[0] + u[1] * v[1] + u[2] * v[2]; };
    const R d1 = dot(ab, ap), d2 = dot(ac, ap);
    R v, w;
    if (d1 <= (R)0 && d2 <= (R)0) { v = 0; w = 0; }
    else {
        const R d3 = dot(ab, bp), d4 = dot(ac, bp);
        const R d5 = dot(ab, cp), d6 = dot(ac, cp);
        const R vc = d1 * d4 - d3 * d2;
        const R vb = d5 * d2 - d1 * d6;
        const R va = d3 * d6 - d5 * d4;
        if (d3 >= (R)0 && d4 <= d3) { v = 1; w = 0; }
        else if (vc <= (R)0 && d1 >= (R)0 && d3 <= (R)0) { v = d1 / (d1 - d3); w = 0; }
        else if (d6 >= (R)0 && d5 <= d6) { v = 0; w = 1; }
        else if (vb <= (R)0 && d2 >= (R)0 && d6 <= (R)0) { v = 0; w = d2 / (d2 - d6); }
        else if (va <= (R)0 && (d4 - d3) >= (R)0 && (d5 - d6) >= (R)0) {
            w = (d4 - d3) / ((d4 - d3) + (d5 - d6));
            v = (R)1 - w;
        } else {
            const R den = (R)1 / (va + vb + vc);
            v = vb * den;
            w = vc * den;
        }
    }
    bary[0] = (R)1 - v - w;
    bary[1] = v;
    bary[2] = w;
    R d2s = 0;
    for (int i = 0; i < 3; ++i) {
        const R q = ap[i] - v * ab[i] - w * ac[i];
        d2s += q * q;
    }
    return d2s;
}

// x <= 0 and x >= 0 of a number that is no NaN, on the integer pipe for
// doubles (a -0 counts as below 0 in ge0: a region's boundary, either side of
// which gives the same point).
__device__ __forceinline__ bool le0(float x) { return x <= 0.0f; }
__device__ __forceinline__ bool ge0(float x) { return x >= 0.0f; }
__device__ __forceinline__ bool le0(double x) { return __double_as_longlong(x) <= 0; }
__device__ __forceinline__ bool ge0(double x) { return __double2hiint(x) >= 0; }
__device__ __forceinline__ bool finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool is0(float x) { return x == 0.0f; }
__device__ __forceinline__ bool is0(double x) { return (__double_as_longlong(x) << 1) == 0; }

// Barycentrics (v of b, w of c) of the point of the triangle (0, b, c) closest
// to P, by the same region tests as closest_tri with the dot products
// relative to vertex a: bp = P - b and cp = P - c enter through
// ab . bp = ab . P - ab . ab and so on. Vertices at one place (the chosen
// region's denominator is 0): the closest point of the longer of ab and ac.
template <typename R>
__device__ __forceinline__ void closest_rel(const R P[3], const R b[3], const R c[3], R bb, R bc, R cc, R& v, R& w) {
    const R d1 = b[0] * P[0] + b[1] * P[1] + b[2] * P[2];
    const R d2 = c[0] * P[0] + c[1] * P[1] + c[2] * P[2];
    if (le0(d1) && le0(d2)) { v = 0; w = 0; return; }
    const R d3 = d1 - bb, d4 = d2 - bc, d5 = d1 - bc, d6 = d2 - cc;
    const R d43 = d4 - d3, d56 = d5 - d6;
    if (ge0(d3) && le0(d43)) { v = 1; w = 0; return; }
    if (ge0(d6) && le0(d56)) { v = 0; w = 1; return; }
    const R vc = d1 * d4 - d3 * d2;
    const R vb = d5 * d2 - d1 * d6;
    const R va = d3 * d6 - d5 * d4;
    // one division for all remaining regions: an edge's or the face's parameter
    const bool e_ab = le0(vc) && ge0(d1) && le0(d3);
    const bool e_ac = !e_ab && le0(vb) && ge0(d2) && le0(d6);
    // (d43 + d56 = |c - b|^2: with both 0, va is rounding)
    const bool e_bc = !e_ab && !e_ac && (le0(va) || (is0(d43) && is0(d56))) && ge0(d43) && ge0(d56);
    const R den = e_ab ? d1 - d3 : e_ac ? d2 - d6 : e_bc ? d43 + d56 : va + vb + vc;
    if (is0(den)) {
        const bool ac = cc >= bb;
        const R len = ac ? cc : bb;
        const R p = len > (R)0 ? fmin(fmax((ac ? d2 : d1) / len, (R)0), (R)1) : (R)0;
        v = ac ? (R)0 : p;
        w = ac ? p : (R)0;
        return;
    }
    const R q = (R)1 / den;
    if (e_ab) { v = d1 * q; w = 0; }
    else if (e_ac) { v = 0; w = d2 * q; }
    else if (e_bc) { w = d43 * q; v = (R)1 - w; }
    else { v = vb * q; w = vc * q; }
}

// Whether the FP32 bounds of the FP64 walks hold for a triangle: big the
// largest component of its edges' cross product, l2 its longest edge squared,
// len the size of the coordinates. They take the triangle to lie in the plane of
// its normal, and the exact test to find its distance to 1e-5 of len. Both need
// an area: with the rounding of nearly parallel edges (or coincident vertices,
// 0 / 0) the normal points anywhere and the exact test's weights are rounding
// too, or no numbers. A height of at least 1/1000 of the longest edge leaves
// the exact test an error of 1e-10 len^2 / edge. FP32 squares of the
// coordinates must not leave the range either. No comparison holds for a NaN.
__device__ __forceinline__ bool has_plane(float big, float l2, float len) {
    return big >= 6e-4f * l2 && l2 > 1e-30f && len > 1e-15f && len < 1e15f;
}

// Box and pair-test geometry of triangle t, axis r = 0..2 by lanes 4 q + r of
// a warp (lane 4 q + 3 only takes part in the shuffles): the FP64 chain of a
// lane is a third of a triangle's. ok: t is a triangle of the mesh. (The node
// positions come from the wing frame: other threads of the launch write xg.)
template <typename T>
__device__ __forceinline__ void tri_setup(const MaskWs& m, const MaskArgs& a, int t, int r, bool ok, double reach) {
    const unsigned all = 0xffffffffu;
    const int ax = r < 3 ? r : 0, l0 = (threadIdx.x & 31) & ~3;
    int id[3] = {0, 0, 0};
    bool good = ok;
    if (ok) {
        for (int v = 0; v < 3; ++v) {
            id[v] = a.tri[3 * t + v];
            good = good && id[v] >= 0 && id[v] < a.n_nodes;
        }
        if (!good) m.cnt[4] = 1;
    }
    double X[3] = {0.0, 0.0, 0.0};
    if (good)
        for (int v = 0; v < 3; ++v) {
            const double* x = a.xw + 3 * (size_t)id[v];
            double s = a.XO[ax];
            for (int c = 0; c < 3; ++c) s += a.R[3 * ax + c] * x[c];
            X[v] = s;
        }
    const double b = X[1] - X[0], c = X[2] - X[0];
    const T tb = (T)b, tc = (T)c;
    // edge components of all three axes from the lanes of this triangle, and
    // as floats (converted once per lane: a conversion is an FP64 instruction)
    const float ob = (float)tb, oc = (float)tc;
    T vb[3], vc[3];
    float fb[3], fc[3];
    for (int q = 0; q < 3; ++q) {
        vb[q] = __shfl_sync(all, tb, l0 + q);
        vc[q] = __shfl_sync(all, tc, l0 + q);
        fb[q] = __shfl_sync(all, ob, l0 + q);
        fc[q] = __shfl_sync(all, oc, l0 + q);
    }
    if (!ok || r == 3) return;
    TriGeo<T>& g = *reinterpret_cast<TriGeo<T>*>(m.geo + (size_t)t * kTriGeoBytes);
    int i0 = 0, e = 0, ca = 0;
    T f = (T)0;
    // a vertex that is no number has no box, so no pair (fmin and fmax would
    // leave it out, and with all three the box would be the whole grid)
    if (good && finite(X[0]) && finite(X[1]) && finite(X[2])) {
        double l = ceil((fmin(X[0], fmin(X[1], X[2])) - reach) * a.inv_dx);
        double h = floor((fmax(X[0], fmax(X[1], X[2])) + reach) * a.inv_dx);
        l = fmax(l, ax == 0 ? (double)a.x_lo : 0.0);
        h = fmin(h, ax == 0 ? (double)(a.x_hi - 1) : (double)((ax == 2 ? a.nz : a.n) - 1));
        i0 = (int)l;
        e = h >= l ? (int)(h - l) + 1 : 0;
        const double cr = floor(X[0] * a.inv_dx);
        ca = (int)cr;
        f = (T)(X[0] - cr * a.dx);
    }
    g.i0[r] = i0;
    g.e[r] = e;
    g.ca[r] = ca;
    g.f[r] = f;
    g.b[r] = tb;
    g.c[r] = tc;
    g.m[r] = (ob + oc) * (1.0f / 3.0f);
    if (r == 0) {
        g.bb = vb[0] * vb[0] + vb[1] * vb[1] + vb[2] * vb[2];
    } else if (r == 1) {
        g.bc = vb[0] * vc[0] + vb[1] * vc[1] + vb[2] * vc[2];
        // sphere about the centroid
        float da = 0.0f, db = 0.0f, dc = 0.0f;
        for (int q = 0; q < 3; ++q) {
            const float mq = (fb[q] + fc[q]) * (1.0f / 3.0f);
            da += mq * mq;
            db += (fb[q] - mq) * (fb[q] - mq);
            dc += (fc[q] - mq) * (fc[q] - mq);
        }
        g.r = sqrtf(fmaxf(da, fmaxf(db, dc))) * 1.00001f;
    } else {
        g.cc = vc[0] * vc[0] + vc[1] * vc[1] + vc[2] * vc[2];
        if constexpr (sizeof(T) == 8) {   // unit normal (only the FP64 walks use it)
            const float n[3] = {(float)(vb[1] * vc[2] - vb[2] * vc[1]), (float)(vb[2] * vc[0] - vb[0] * vc[2]),
                                (float)(vb[0] * vc[1] - vb[1] * vc[0])};
            float l2 = 0.0f, bb = 0.0f, cc = 0.0f;   // squared edge lengths
            for (int q = 0; q < 3; ++q) {
                bb += fb[q] * fb[q];
                cc += fc[q] * fc[q];
                l2 += (fb[q] - fc[q]) * (fb[q] - fc[q]);
            }
            l2 = fmaxf(l2, fmaxf(bb, cc));
            const float big = fmaxf(fabsf(n[0]), fmaxf(fabsf(n[1]), fabsf(n[2])));
            const bool plane = has_plane(big, l2, sqrtf(l2) + (float)reach);
            const float k = plane ? 1.0f / big : 0.0f;
            const float x = n[0] * k, y = n[1] * k, z = n[2] * k, u = plane ? rsqrtf(x * x + y * y + z * z) : 0.0f;
            g.nrm[0] = x * u;
            g.nrm[1] = y * u;
            g.nrm[2] = z * u;
        }
    }
}

// First kernel of a call: zero chi/u_s and reset the key and winner of the
// points the previous call touched (list `par`), clear the line flags
// (n^2 bytes, 16-byte aligned), reset the other list's count, the global
// node positions X_O + R x^(w) (double), and (BAND) the triangles' boxes and
// geometry. The triangles start at the last thread (four each) and the nodes
// at the first, so that as few warps as possible have both FP64 chains.
template <typename T, bool BAND>
__global__ void k_mask_prepare(MaskWs m, MaskArgs a, int par, T* chi, T* us, uint8_t* flag, size_t n3, size_t nflag,
                               double reach) {
    pdl_wait();
    const unsigned long long tid = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned long long nth = (unsigned long long)gridDim.x * blockDim.x;
    if (tid == 0) m.cnt[par ^ 1] = 0;
    if (tid < (unsigned long long)a.n_nodes) {
        const int i = (int)tid;
        for (int r = 0; r < 3; ++r) {
            double s = a.XO[r], v = 0.0;
            for (int c = 0; c < 3; ++c) {
                s += a.R[3 * r + c] * a.xw[3 * i + c];
                v += a.R[3 * r + c] * a.vw[3 * i + c];
            }
            m.xg[3 * i + r] = s;
            m.vg[3 * i + r] = v;
        }
    }
    if constexpr (BAND) {
        // thread u from the end: whole warps, four lanes per triangle
        const unsigned long long w = (nth - 1 - tid) >> 5;
        const unsigned long long t = 8 * w + ((threadIdx.x & 31) >> 2);
        if (8 * w < (unsigned long long)a.n_tri)   // uniform in the warp
            tri_setup<T>(m, a, (int)t, threadIdx.x & 3, t < (unsigned long long)a.n_tri, reach);
    }
    uint4* f4 = reinterpret_cast<uint4*>(flag);
    for (unsigned long long i = tid; i < nflag / 16; i += nth) f4[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < nflag % 16) flag[nflag / 16 * 16 + tid] = 0;
    const unsigned long long cnt = m.cnt[par];
    const uint32_t* L = par ? m.list[1] : m.list[0];
    for (unsigned long long i = tid; i < cnt; i += nth) {
        const uint32_t p = L[i];
        m.key[p] = ~0ull;
        m.win[p] = 0x7fffffff;
        chi[p] = (T)0;
        for (int c = 0; c < 3; ++c) us[c * n3 + p] = (T)0;
    }
}

// Tolerance of near-ties of squared distances (FP64): 4 units in the last
// place of the distance (the same pair recomputed may round differently).
__device__ __forceinline__ double tie_limit(double d2) { return d2 + (d2 * 1.8e-15 + 1e-300); }

// Bits of the double equal to a normal float > 0, and the float at or just
// below a double given by its bits (0 below the float range, its end above):
// on the integer pipe, a conversion takes 64 cycles like any FP64 instruction.
__device__ __forceinline__ unsigned long long widen(float x) {
    return ((unsigned long long)__float_as_uint(x) << 29) + (896ull << 52);
}
__device__ __forceinline__ float narrow(unsigned long long bits) {
    const long long e = (long long)(bits >> 29) - (896ll << 23);
    return __int_as_float(e < 0 ? 0 : e > 0x7f7fffffll ? 0x7f7fffff : (int)e);
}

// Warp (t, part) of wpt per triangle: points 32 part .. 32 part + 31 of
// triangle t's box, and on by 32 wpt.
static constexpr int kPairThreads = 256;
enum PairWalk { kPairOne, kPairBound, kPairLeast, kPairTies };
template <typename T, int WALK>
__global__ void __launch_bounds__(kPairThreads) k_mask_pairs(MaskWs m, MaskArgs a, int par, int wpt) {
    pdl_wait();
    const uint32_t warp = (blockIdx.x * (uint32_t)kPairThreads + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int t = (int)(warp / (uint32_t)wpt);
    if (t >= a.n_tri) return;   // whole warps leave together
    const TriGeo<T> g = *reinterpret_cast<const TriGeo<T>*>(m.geo + (size_t)t * kTriGeoBytes);
    const uint32_t ej = (uint32_t)g.e[1], ek = (uint32_t)g.e[2], cnt = (uint32_t)g.e[0] * ej * ek;
    const uint32_t l1 = 32u * (warp % (uint32_t)wpt), step = 32u * (uint32_t)wpt;
    const double reach = a.tw + a.h;
    uint32_t* const list = par ? m.list[1] : m.list[0];
    auto place = [&](uint32_t l, int& i, int& j, int& k) {
        const uint32_t q = l / ek;
        k = g.i0[2] + (int)(l - q * ek);
        i = (int)(q / ej);
        j = g.i0[1] + (int)(q - (uint32_t)i * ej);
        i += g.i0[0];
    };
    auto index = [&](int i, int j, int k) { return ((uint32_t)i * (uint32_t)a.n + (uint32_t)j) * (uint32_t)a.nz + (uint32_t)k; };
    auto dist2 = [&](int i, int j, int k) -> T {
        const T dx = (T)a.dx;
        const T P[3] = {(T)(i - g.ca[0]) * dx - g.f[0], (T)(j - g.ca[1]) * dx - g.f[1], (T)(k - g.ca[2]) * dx - g.f[2]};
        T v, w, s = (T)0;
        closest_rel<T>(P, g.b, g.c, g.bb, g.bc, g.cc, v, w);
        for (int r = 0; r < 3; ++r) {
            const T q = P[r] - v * g.b[r] - w * g.c[r];
            s += q * q;
        }
        return s;
    };
    auto offer = [&](uint32_t p, unsigned long long key) {
        if (atomicMin(&m.key[p], key) == ~0ull) list[atomicAdd(&m.cnt[par], 1ull)] = p;
    };
    if constexpr (WALK == kPairOne) {
        const T reach2 = (T)(reach * reach);
        for (uint32_t l = l1 + lane; l < cnt; l += step) {
            int i, j, k;
            place(l, i, j, k);
            const T d2 = dist2(i, j, k);
            if (d2 < reach2) offer(index(i, j, k), ((unsigned long long)__float_as_uint((float)d2) << 32) | (uint32_t)t);
        }
    } else {
        // FP32 bounds of a pair's distance: the triangle lies in the disc of
        // radius r about m in its plane, and a point of it with clamped
        // barycentrics is at least as far as the closest one. Both are
        // rounded outwards by err, some thirty times the rounding of the
        // coordinates (at most 2 r + reach + a cell, 1.2e-7 of that). A
        // triangle without a plane bounds nothing: its points go to the list
        // with an infinite key and every pair of its box to the exact test.
        const bool plane = g.nrm[0] != 0.0f || g.nrm[1] != 0.0f || g.nrm[2] != 0.0f;
        const float fdx = (float)a.dx, freach = (float)reach, err = 1e-5f * (g.r + freach + fdx);
        const float ff[3] = {(float)g.f[0], (float)g.f[1], (float)g.f[2]};
        auto at = [&](int i, int j, int k, float* P) {
            P[0] = (float)(i - g.ca[0]) * fdx - ff[0];
            P[1] = (float)(j - g.ca[1]) * fdx - ff[1];
            P[2] = (float)(k - g.ca[2]) * fdx - ff[2];
        };
        auto lower = [&](const float* P) {
            if (!plane) return 0.0f;
            const float x = P[0] - g.m[0], y = P[1] - g.m[1], z = P[2] - g.m[2];
            const float h = x * g.nrm[0] + y * g.nrm[1] + z * g.nrm[2], h2 = h * h;
            const float in = fmaxf(sqrtf(fmaxf(x * x + y * y + z * z - h2, 0.0f)) - g.r - err, 0.0f);
            return fmaxf(sqrtf(h2 + in * in) - err, 0.0f);
        };
        if constexpr (WALK == kPairBound) {
            const float b[3] = {(float)g.b[0], (float)g.b[1], (float)g.b[2]}, c[3] = {(float)g.c[0], (float)g.c[1], (float)g.c[2]};
            for (uint32_t l = l1 + lane; l < cnt; l += step) {
                int i, j, k;
                place(l, i, j, k);
                float P[3], v, w, s = 0.0f;
                at(i, j, k, P);
                if (lower(P) > freach) continue;
                if (!plane) {
                    offer(index(i, j, k), 0x7ff0000000000000ull);
                    continue;
                }
                closest_rel<float>(P, b, c, (float)g.bb, (float)g.bc, (float)g.cc, v, w);
                v = fminf(fmaxf(v, 0.0f), 1.0f);
                w = fminf(fmaxf(w, 0.0f), 1.0f - v);
                for (int r = 0; r < 3; ++r) {
                    const float q = P[r] - v * b[r] - w * c[r];
                    s += q * q;
                }
                const float up = sqrtf(s) + err;
                offer(index(i, j, k), widen(fmaxf(up * up * 1.00001f, 1e-37f)));
            }
        } else {
            const double reach2 = reach * reach;
            // pairs that the bounds leave wait in the warp's queue until 32 are there
            __shared__ uint32_t queue[kPairThreads / 32][64];
            uint32_t* const Q = queue[threadIdx.x >> 5];
            int nq = 0;
            auto test = [&](bool on, uint32_t l) {
                if (!on) return;
                int i, j, k;
                place(l, i, j, k);
                const uint32_t p = index(i, j, k);
                const double d2 = (double)dist2(i, j, k);
                if (!(d2 < reach2)) return;
                if constexpr (WALK == kPairTies) {
                    if (d2 <= tie_limit(__longlong_as_double((long long)m.key[p]))) atomicMin(&m.win[p], t);
                } else {
                    atomicMin(&m.key[p], (unsigned long long)__double_as_longlong(d2));
                }
            };
            for (uint32_t l0 = l1; l0 < cnt; l0 += step) {
                const uint32_t l = l0 + lane;
                bool in = l < cnt;
                if (in) {
                    int i, j, k;
                    place(l, i, j, k);
                    float P[3];
                    at(i, j, k, P);
                    const float lo = lower(P);
                    // at most the least distance so far, with the tie's margin
                    const unsigned long long key = __ldcg(&m.key[index(i, j, k)]);
                    in = lo <= freach && lo * lo <= narrow(key) * 1.0001f + 2e-37f;
                }
                const unsigned b = __ballot_sync(0xffffffffu, in);
                if (in) Q[nq + __popc(b & ((1u << lane) - 1u))] = l;
                nq += __popc(b);
                __syncwarp();
                if (nq >= 32) {
                    nq -= 32;
                    test(true, Q[nq + lane]);
                    __syncwarp();
                }
            }
            test(lane < nq, lane < nq ? Q[lane] : 0u);
        }
    }
}

// sin(pi s), |s| <= 1/2: its series to s^21 (the next term is below 1e-17
// there); half the FP64 instructions of cospi with its range reduction.
__device__ __forceinline__ double sin_pi_half(double s) {
    const double q = s * s;
    double r = 5.39266466260812895e-10;
    r = fma(r, q, -2.29484289972698730e-08);
    r = fma(r, q, 7.95205400147551261e-07);
    r = fma(r, q, -2.19153534478302173e-05);
    r = fma(r, q, 4.66302805767612554e-04);
    r = fma(r, q, -7.37043094571435044e-03);
    r = fma(r, q, 8.21458866111282326e-02);
    r = fma(r, q, -5.99264529320792105e-01);
    r = fma(r, q, 2.55016403987734552e+00);
    r = fma(r, q, -5.16771278004997026e+00);
    r = fma(r, q, 3.14159265358979312e+00);
    return r * s;
}

__device__ __forceinline__ double chi_profile(double d, double tw, double h, int profile) {
    if (profile == 1) return 0.5 * (1.0 - tanh((d - tw) / h));
    if (d <= tw - h) return 1.0;
    if (d >= tw + h) return 0.0;
    return 0.5 - 0.5 * sin_pi_half((d - tw) * (0.5 / h));   // = (1 + cos(pi (d - tw + h) / (2 h))) / 2
}

// chi and u_s at grid point p from triangle t (double throughout).
template <typename T>
__device__ __forceinline__ void eval_point(const MaskWs& m, const MaskArgs& a, uint32_t p, int t, T* chi, T* us,
                                           uint8_t* flag) {
    const uint32_t un = (uint32_t)a.n, unz = (uint32_t)a.nz;
    const size_t n3 = (size_t)un * un * unz;
    const uint32_t line = p / unz, i = line / un;
    const int k = (int)(p - line * unz), j = (int)(line - i * un);
    const int id[3] = {a.tri[3 * t], a.tri[3 * t + 1], a.tri[3 * t + 2]};
    const double X[3] = {(int)i * a.dx, j * a.dx, k * a.dx};
    double P[3], b[3], c[3], bb = 0.0, bc = 0.0, cc = 0.0;
    for (int r = 0; r < 3; ++r) {
        const double x0 = m.xg[3 * id[0] + r];
        P[r] = X[r] - x0;
        b[r] = m.xg[3 * id[1] + r] - x0;
        c[r] = m.xg[3 * id[2] + r] - x0;
        bb += b[r] * b[r];
        bc += b[r] * c[r];
        cc += c[r] * c[r];
    }
    double v, w, d2 = 0.0;
    closest_rel<double>(P, b, c, bb, bc, cc, v, w);
    for (int r = 0; r < 3; ++r) {
        const double q = P[r] - v * b[r] - w * c[r];
        d2 += q * q;
    }
    const double chi_p = chi_profile(sqrt(d2), a.tw, a.h, a.profile);
    chi[p] = (T)chi_p;
    if (chi_p > 0.0 || a.profile == 1) {
        // u_s = V_O + Omega x (x - X_O) + sum beta R v
        const double u = 1.0 - v - w;
        const double rr[3] = {X[0] - a.XO[0], X[1] - a.XO[1], X[2] - a.XO[2]};
        for (int r = 0; r < 3; ++r) {
            const int r1 = (r + 1) % 3, r2 = (r + 2) % 3;
            double g = a.VO[r] + a.Om[r1] * rr[r2] - a.Om[r2] * rr[r1];
            g += u * m.vg[3 * id[0] + r] + v * m.vg[3 * id[1] + r] + w * m.vg[3 * id[2] + r];
            us[r * n3 + p] = (T)g;
        }
        if (chi_p > 0.0) flag[line] = 1;
    }
}

template <typename T>
__global__ void k_mask_eval(MaskWs m, MaskArgs a, int par, T* chi, T* us, uint8_t* flag) {
    pdl_wait();
    const unsigned long long cnt = m.cnt[par];
    const uint32_t* const list = par ? m.list[1] : m.list[0];
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t p = list[i];
        int t;
        if constexpr (sizeof(T) == 4) {   // the winner is the key's low word; kept for the VJP
            t = (int)(uint32_t)m.key[p];
            m.win[p] = t;
        } else {
            t = m.win[p];
        }
        if (t >= 0 && t < a.n_tri) eval_point<T>(m, a, p, t, chi, us, flag);
    }
}

// Dense (tanh) profile: every point against every triangle in index order.
template <typename T>
__global__ void k_mask_dense(MaskWs m, MaskArgs a, T* chi, T* us, uint8_t* flag) {
    pdl_wait();
    const size_t n = a.n, nz = a.nz, n3 = n * n * nz;
    for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < n3; p += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(p % nz), j = (int)((p / nz) % n), i = (int)(p / (n * nz));
        if (i < a.x_lo || i >= a.x_hi) continue;
        T best = (T)3.0e38;
        int bt = 0;
        for (int t = 0; t < a.n_tri; ++t) {
            const int ia = a.tri[3 * t], ib = a.tri[3 * t + 1], ic = a.tri[3 * t + 2];
            if (ia < 0 || ib < 0 || ic < 0 || ia >= a.n_nodes || ib >= a.n_nodes || ic >= a.n_nodes) {
                if (p == 0) m.cnt[4] = 1;
                continue;
            }
            const double ax = m.xg[3 * ia], ay = m.xg[3 * ia + 1], az = m.xg[3 * ia + 2];
            T P[3] = {(T)(i * a.dx - ax), (T)(j * a.dx - ay), (T)(k * a.dx - az)};
            T A0[3] = {(T)0, (T)0, (T)0};
            T B0[3] = {(T)(m.xg[3 * ib] - ax), (T)(m.xg[3 * ib + 1] - ay), (T)(m.xg[3 * ib + 2] - az)};
            T C0[3] = {(T)(m.xg[3 * ic] - ax), (T)(m.xg[3 * ic + 1] - ay), (T)(m.xg[3 * ic + 2] - az)};
            T bary[3];
            const T d = sqrt(closest_tri<T>(P, A0, B0, C0, bary));
            if (d < best) { best = d; bt = t; }
        }
        eval_point<T>(m, a, (uint32_t)p, bt, chi, us, flag);
    }
}

// Host driver (in ps_api.cu). `par` is the index of the touched list the
// previous call filled; the call clears those points, fills the other list
// and returns its index in *par_out. `init` resets every key (first call);
// `dense_dirty` zeroes chi/u_s everywhere first (after a dense mask).
template <typename T>
cudaError_t rasterise(const MaskArgs& a, void* chi, void* us, uint8_t* flag, unsigned char* ws, int par, bool init,
                      bool dense_dirty, cudaStream_t s, int* par_out);

}  // namespace ps
