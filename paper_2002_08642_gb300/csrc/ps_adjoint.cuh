// ps_adjoint.cuh -- discrete adjoint of one time step and of the wing mask
// rasteriser (no counterpart in the paper; the exact transpose of the step's
// operations, for objectives J = sum_n (a_n . F^n + b_n . M^n)).
//
// Conventions: U holds Fourier coefficients c (u = inverse(c), no scaling;
// forward(u) = DFT(u) / n^3). Adjoint variables live on the same compact
// spectral layout with the inner product Re sum w conj(x) y (w = 1 on the
// kz = 0 plane, 2 elsewhere), under which inverse* = n^3 forward and
// forward* = inverse / n^3; truncation, projection, E and i k x are
// self-adjoint mode by mode. Per reversed step n (lam = dL/du^{n+1},
// mu = dL/dH^{n+1}):
//   Gbar = a1 lam + mu  (a1 = 1.5 dt E, or dt E for the Euler start step)
//   G    = P Gbar        -> nbar = inverse(G) / n^3       (physical)
//   lam' = E lam,  mu' = -0.5 dt E^2 lam  (0 for the start step)
//   ubar = omega x nbar - (chi/eta) nbar + (dx^3/eta) chi (a + b x r)
//   wbar = nbar x u
//   dJ/dchi = -(1/eta) nbar . (u - us) + (dx^3/eta) (a + b x r) . (u - us)
//   dJ/dus  = (chi/eta) nbar - (dx^3/eta) chi (a + b x r)
//   lam' += n^3 [forward(ubar) + i k x forward(wbar)]
#pragma once
#include "ps_adjoint_z.cuh"
#include "ps_kernels.cuh"

namespace ps {

// Spectral part: G = P (a1 lam + mu). (The x-forward pass at the end of the
// reversed step updates lam and mu.)
template <typename T>
__global__ void k_adj_spec(KP kp, const cplx<T>* __restrict__ lam, const cplx<T>* __restrict__ mu, cplx<T>* __restrict__ G,
                           const T* __restrict__ Ex, const T* __restrict__ Ez, int first) {
    pdl_wait();
    using C2 = cplx<T>;
    const int K = kp.K, Kz = kp.Kz, Kzp = kp.Kzp, mm = kp.mmax;
    const size_t FS = (size_t)K * K * Kzp;
    const size_t tot = (size_t)K * K * Kz;
    const T dt = (T)kp.dt, s = (T)kp.ks, sz = (T)kp.ksz;
    // 32-bit index arithmetic: K^2 Kz < 2^27 for every grid the library builds
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < (uint32_t)tot; i += gridDim.x * blockDim.x) {
        const int cz = (int)(i % (uint32_t)Kz);
        const uint32_t r = i / (uint32_t)Kz;
        const int cx = (int)(r % (uint32_t)K), cy = (int)(r / (uint32_t)K);
        const size_t o = ((size_t)cy * K + cx) * Kzp + cz;
        const T E = Ex[cx] * Ex[cy] * Ez[cz];
        const T a1 = first ? dt * E : (T)1.5 * dt * E;
        C2 g[3];
        for (int f = 0; f < 3; ++f) {
            const C2 l = lam[f * FS + o], m = mu[f * FS + o];
            g[f] = cmk<C2>(a1 * l.x + m.x, a1 * l.y + m.y);
        }
        const int mx = cmode_of(cx, mm, K), my = cmode_of(cy, mm, K);
        const T kx = s * (T)mx, ky = s * (T)my, kz = sz * (T)cz;
        if (mx == 0 && my == 0 && cz == 0) {
            if (!kp.mean_free) g[0] = g[1] = g[2] = cmk<C2>((T)0, (T)0);
        } else {
            const T ik2 = (T)1 / (kx * kx + ky * ky + kz * kz);
            const T dr = (kx * g[0].x + ky * g[1].x + kz * g[2].x) * ik2;
            const T di = (kx * g[0].y + ky * g[1].y + kz * g[2].y) * ik2;
            g[0].x -= kx * dr; g[0].y -= kx * di;
            g[1].x -= ky * dr; g[1].y -= ky * di;
            g[2].x -= kz * dr; g[2].y -= kz * di;
        }
        for (int f = 0; f < 3; ++f) G[f * FS + o] = g[f];
    }
}

// ------------------------------------------------ rasteriser VJP
__device__ __forceinline__ double chi_profile_d(double d, double tw, double h, int profile) {
    if (profile == 1) {
        const double t = tanh((d - tw) / h);
        return -0.5 * (1.0 - t * t) / h;
    }
    if (d <= tw - h || d >= tw + h) return 0.0;
    const double t = (d - tw + h) * (0.5 / h);   // -(pi / 4 h) sin(pi t), 0 < t < 1
    return -0.25 * M_PI / h * sin_pi_half(t <= 0.5 ? t : 1.0 - t);
}

// One grid point p with closest triangle t: dJ/dX (global vertex positions)
// accumulated into gX with atomics. The closest triangle is held fixed; the
// distance derivative is -beta_v (p - q)/delta (envelope theorem), the
// barycentric weights are differentiated on their active face.
// One chain of FP64 instructions per point (64 cycles each): positions
// relative to vertex 0, the node velocities rotated beforehand, an edge's two
// vertices picked by selects instead of indexed local arrays (GB300, wing at
// 64^3 FP64: 48 -> 27 us per call).
template <typename T>
__device__ void vjp_point(const MaskWs& m, const MaskArgs& a, uint32_t p, int t, const T* __restrict__ gchi,
                          const T* __restrict__ gus, const T* __restrict__ chi, double* __restrict__ gX) {
    const uint32_t un = (uint32_t)a.n, unz = (uint32_t)a.nz, line = p / unz, i = line / un;
    const size_t n3 = (size_t)un * un * unz;
    const double X[3] = {(int)i * a.dx, (int)(line - i * un) * a.dx, (int)(p - line * unz) * a.dx};
    const int id[3] = {a.tri[3 * t], a.tri[3 * t + 1], a.tri[3 * t + 2]};
    double P[3], e1[3], e2[3], m00 = 0.0, m01 = 0.0, m11 = 0.0;   // point and vertices 1, 2 relative to vertex 0
    for (int r = 0; r < 3; ++r) {
        const double x0 = m.xg[3 * id[0] + r];
        P[r] = X[r] - x0;
        e1[r] = m.xg[3 * id[1] + r] - x0;
        e2[r] = m.xg[3 * id[2] + r] - x0;
        m00 += e1[r] * e1[r];
        m01 += e1[r] * e2[r];
        m11 += e2[r] * e2[r];
    }
    double s_, t_, q[3], d2 = 0.0;
    closest_rel<double>(P, e1, e2, m00, m01, m11, s_, t_);
    const double u_ = 1.0 - s_ - t_;
    for (int r = 0; r < 3; ++r) {
        q[r] = P[r] - s_ * e1[r] - t_ * e2[r];
        d2 += q[r] * q[r];
    }
    const double d = sqrt(d2);
    double acc[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    const double cb = (double)gchi[p];
    if (d > 0.0 && cb != 0.0) {
        const double gd = -cb * chi_profile_d(d, a.tw, a.h, a.profile) / d;
        for (int r = 0; r < 3; ++r) {
            const double f = gd * q[r];
            acc[0][r] = f * u_;
            acc[1][r] = f * s_;
            acc[2][r] = f * t_;
        }
    }
    const bool has_us = (a.profile == 1) || (double)chi[p] > 0.0;
    if (has_us) {
        double g[3] = {0.0, 0.0, 0.0};   // dJ/dbeta_v = (dJ/du_s) . (R vw_v)
        for (int r = 0; r < 3; ++r) {
            const double ub = (double)gus[r * n3 + p];
            for (int v = 0; v < 3; ++v) g[v] += ub * m.vg[3 * id[v] + r];
        }
        const bool on0 = u_ > 1e-12, on1 = s_ > 1e-12, on2 = t_ > 1e-12;
        const int na = (int)on0 + (int)on1 + (int)on2;
        if (na == 2) {   // edge from vertex iu to iv > iu: iu = 0 if on0 else 1, iv = 2 if on2 else 1
            double e[3], pu[3], dd = 0.0, nn = 0.0;
            for (int r = 0; r < 3; ++r) {
                const double xu = on0 ? 0.0 : e1[r], xv = on2 ? e2[r] : e1[r];
                e[r] = xv - xu;
                pu[r] = P[r] - xu;
                dd += e[r] * e[r];
                nn += pu[r] * e[r];
            }
            const double gt = ((on2 ? g[2] : g[1]) - (on0 ? g[0] : g[1])) / (dd * dd), n2 = 2.0 * nn;
            for (int r = 0; r < 3; ++r) {
                const double fv = gt * (pu[r] * dd - n2 * e[r]);
                const double fu = gt * (n2 * e[r] - (e[r] + pu[r]) * dd);
                if (on0) acc[0][r] += fu; else acc[1][r] += fu;
                if (on2) acc[2][r] += fv; else acc[1][r] += fv;
            }
        } else if (na == 3) {
            const double g0 = g[1] - g[0], g1 = g[2] - g[0];
            const double idet = 1.0 / (m00 * m11 - m01 * m01);
            const double z0 = (m11 * g0 - m01 * g1) * idet, z1 = (m00 * g1 - m01 * g0) * idet;
            for (int r = 0; r < 3; ++r) {
                const double cdd = z0 * e1[r] + z1 * e2[r];
                const double ce0 = z0 * P[r] - (z0 * (2.0 * s_ * e1[r] + t_ * e2[r]) + z1 * (s_ * e2[r]));
                const double ce1 = z1 * P[r] - (z0 * (t_ * e1[r]) + z1 * (s_ * e1[r] + 2.0 * t_ * e2[r]));
                acc[0][r] += -cdd - ce0 - ce1;
                acc[1][r] += ce0;
                acc[2][r] += ce1;
            }
        }
    }
    for (int v = 0; v < 3; ++v)
        for (int r = 0; r < 3; ++r)
            if (acc[v][r] != 0.0) atomicAdd(&gX[3 * id[v] + r], acc[v][r]);
}

template <typename T>
__global__ void k_mask_vjp_list(MaskWs m, MaskArgs a, int par, const T* __restrict__ gchi,
                                const T* __restrict__ gus, const T* __restrict__ chi, double* __restrict__ gX) {
    pdl_wait();
    const unsigned long long cnt = m.cnt[par];
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t p = m.list[par][i];
        const int t = m.win[p];
        if (t >= 0 && t < a.n_tri) vjp_point<T>(m, a, p, t, gchi, gus, chi, gX);
    }
}

// dense (tanh) profile: the closest triangle is recomputed per point
template <typename T>
__global__ void k_mask_vjp_dense(MaskWs m, MaskArgs a, const T* __restrict__ gchi, const T* __restrict__ gus,
                                 const T* __restrict__ chi, double* __restrict__ gX) {
    pdl_wait();
    const size_t n = a.n, nz = a.nz, n3 = n * n * nz;
    for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < n3; p += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(p % nz), j = (int)((p / nz) % n), i = (int)(p / (n * nz));
        T best = (T)3.0e38;
        int bt = -1;
        for (int t = 0; t < a.n_tri; ++t) {
            const int ia = a.tri[3 * t], ib = a.tri[3 * t + 1], ic = a.tri[3 * t + 2];
            if (ia < 0 || ib < 0 || ic < 0 || ia >= a.n_nodes || ib >= a.n_nodes || ic >= a.n_nodes) continue;
            const double ax = m.xg[3 * ia], ay = m.xg[3 * ia + 1], az = m.xg[3 * ia + 2];
            T P[3] = {(T)(i * a.dx - ax), (T)(j * a.dx - ay), (T)(k * a.dx - az)};
            T A0[3] = {(T)0, (T)0, (T)0};
            T B0[3] = {(T)(m.xg[3 * ib] - ax), (T)(m.xg[3 * ib + 1] - ay), (T)(m.xg[3 * ib + 2] - az)};
            T C0[3] = {(T)(m.xg[3 * ic] - ax), (T)(m.xg[3 * ic + 1] - ay), (T)(m.xg[3 * ic + 2] - az)};
            T bary[3];
            const T d = sqrt(closest_tri<T>(P, A0, B0, C0, bary));
            if (d < best) { best = d; bt = t; }
        }
        if (bt >= 0) vjp_point<T>(m, a, (uint32_t)p, bt, gchi, gus, chi, gX);
    }
}

// grad_xw[v] += R^T gX[v]  (global -> wing frame)
__global__ void k_vjp_to_wing(MaskArgs a, const double* __restrict__ gX, double* __restrict__ gxw) {
    pdl_wait();
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= a.n_nodes) return;
    for (int c = 0; c < 3; ++c) {
        double s = 0.0;
        for (int r = 0; r < 3; ++r) s += a.R[3 * r + c] * gX[3 * v + r];
        gxw[3 * v + c] += s;
    }
}

}  // namespace ps
