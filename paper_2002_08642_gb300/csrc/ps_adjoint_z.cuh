// ps_adjoint_z.cuh -- the z pass of a reversed time step: physical u, omega
// and nbar of a batch of z lines, the pointwise adjoint, and the forward
// transforms of its results, in one kernel (ps_adjoint.cuh has the formulas).
#pragma once
#include "ps_kernels.cuh"

namespace ps {

struct AdjW {
    double a[3], b[3];   // dJ/dF, dJ/dM of this step
    int first;           // reversing the integrating-factor Euler start step
};

// Batches of one line pair, nine thread groups of G threads: groups 3 f + q of
// vector f (0: u, 1: omega, 2: nbar) transform (x + i y) of line 0, of line 1
// (q = 0, 1) and (z of line 0 + i z of line 1) (q = 2); f < 2 also transform
// the results ubar, wbar forward the same way. A complex line never mixes two
// vectors: u and omega, ubar and wbar differ by two orders of magnitude, and
// the rounding of the larger would go into the smaller (dJ/dchi in FP32 was
// off by 1.4e-6 instead of 2.3e-7 with u_z + i omega_x packed).
// For n = 3M the sub-lines lie SUB apart: SUB = 6 mod 16, so that reading
// consecutive z (sub-lines in turn) meets no bank twice.
template <typename T, int N> struct AdjZ {
    using C2 = cplx<T>;
    using GE = Geo<T, N>;
    using S3 = Split3<T, N>;
    static constexpr bool Z3 = S3::on;
    static constexpr bool PAD = Z3 && S3::M % 16 == 0;   // sub-lines on padding groups
    static constexpr int SUB = PAD ? S3::M + S3::M / 16 + ((6 - (S3::M + S3::M / 16)) % 16 + 16) % 16 : 0;
    static constexpr int LP = PAD ? 3 * SUB : N + N / 16 + 1;
    static constexpr int threads = 9 * GE::G;
    static constexpr int smem = (int)sizeof(C2) * (9 * 2 * GE::KZP + 9 * LP + tw_count(N, GE::RM) + 1) + 128;
    // blocks per SM the register budget is sized for: what the shared memory
    // holds, at most about 900 threads (72 registers each)
    static constexpr int fit = (227 * 1024) / (smem + 2048) > 0 ? (227 * 1024) / (smem + 2048) : 1;
    static constexpr int most = 900 / threads > 16 ? 16 : 900 / threads > 0 ? 900 / threads : 1;
    static constexpr int minb = fit < most ? fit : most;
};

// B: u, omega (fields 0..5, z spectral) on entry, ubar, wbar on return (a
// batch's own lines, whose input is in shared memory by then); NB: nbar,
// inverse(G), three z-spectral fields, unscaled. Writes dJ/dchi and dJ/du_s.
// Memory: fifteen z-spectral fields and eight physical ones cross HBM once;
// as separate inverse transforms, pointwise kernel and forward transforms
// thirty more physical fields went out and came back (GB300, 512^3 FP32: three
// inverse, one pointwise and two forward kernels 4.29 ms, this 2.96 ms). It is
// bound by its fifteen line transforms' exchanges through shared memory: at 384 x
// 384 x 192 184 M wavefronts in 0.71 ms, 83 % of the SMs' rate, 37 % of them bank
// conflicts; issue slots 54 %, DRAM 34 %.
template <typename T, int N, int NY = N>
__global__ void __launch_bounds__(AdjZ<T, N>::threads, AdjZ<T, N>::minb)
k_adj_zpass(KP kp, AdjW aw, cplx<T>* __restrict__ B, const cplx<T>* __restrict__ NB, const T* __restrict__ chi,
            const T* __restrict__ us, const uint8_t* __restrict__ flag, T* __restrict__ gchi, T* __restrict__ gus,
            const cplx<T>* __restrict__ twg, int* __restrict__ err) {
    using C2 = cplx<T>;
    using AZ = AdjZ<T, N>;
    using GE = Geo<T, N>;
    using S3 = Split3<T, N>;
    constexpr int G = GE::G, KZP = GE::KZP, LP = AZ::LP, M = S3::M, GM = S3::GM;
    constexpr bool Z3 = AZ::Z3, PAD = AZ::PAD;
    constexpr int SUB = AZ::SUB;
    constexpr int GL = Z3 ? GM : G;
    constexpr bool WS = GL <= 32 && 32 % GL == 0;
    constexpr uint32_t fbytes = (uint32_t)(2 * KZP * sizeof(C2));
    extern __shared__ __align__(16) unsigned char smraw[];
    C2* stage = reinterpret_cast<C2*>(smem_base128(smraw));   // [9][2][KZP]
    if (smem_u32(stage) & 127u) {   // never expected: refuse to start copies
        pdl_wait();
        if (threadIdx.x == 0) atomicExch(err, 2);
        return;
    }
    C2* tiles = stage + 9 * 2 * KZP;   // [9][LP]
    C2* tw = tiles + 9 * LP;
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint8_t sflag[2];
    const int grp = threadIdx.x / G, g = threadIdx.x % G;
    const int Kz = kp.Kz;
    const size_t nlines = (size_t)NY * NY, BS = nlines * KZP, N3 = nlines * N;
    const int nb = (int)(nlines / 2);
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    C2* tw3 = load_tw_split<T, N>(tw, twg, GE::tw_n);
    __syncthreads();
    pdl_wait();
    auto issue = [&](int b) {  // one thread
        fence_proxy_async();
        mbar_arrive_expect_tx(&bar, 9 * fbytes);
#pragma unroll 1
        for (int f = 0; f < 9; ++f)
            bulk_g2s(stage + (size_t)f * 2 * KZP, (f < 6 ? B + f * BS : NB + (f - 6) * BS) + (size_t)b * 2 * KZP, fbytes,
                     &bar);
    };
    if (threadIdx.x == 0 && (int)blockIdx.x < nb) issue(blockIdx.x);
    // constants in T: no double arithmetic per point
    const T inv_eta = (T)kp.inv_eta, invn3 = (T)kp.invn3, dx = (T)kp.dx;
    const T fs = (T)(kp.dx * kp.dx * kp.dx * kp.inv_eta);
    const T a0 = (T)aw.a[0], a1 = (T)aw.a[1], a2 = (T)aw.a[2];
    const T b0 = (T)aw.b[0], b1 = (T)aw.b[1], b2 = (T)aw.b[2];
    // this group's input lines
    const int vec = grp / 3, q = grp % 3;
    const C2* const fa = stage + (q < 2 ? (vec * 3 * 2 + q) * KZP : (vec * 3 + 2) * 2 * KZP);
    const C2* const fb = q < 2 ? fa + 2 * KZP : fa + KZP;
    const int tbase = grp * LP;
    // tile position of z
    auto zpos = [&](int z) { return PAD ? (z % 3) * SUB + z / 3 + ((z / 3) >> 4) : Z3 ? zaddr((z % 3) * M + z / 3, 0, 0) : z + (z >> 4); };
    int it = 0;
    for (int b = blockIdx.x; b < nb; b += gridDim.x, ++it) {
        const bool more = b + (int)gridDim.x < nb;
        const bool ok = mbar_wait(&bar, (uint32_t)(it & 1));
        if (__syncthreads_or(!ok)) {
            // a copy never completed: record it, let it land, stop
            if (threadIdx.x == 0) {
                atomicExch(err, 1);
                mbar_wait(&bar, (uint32_t)(it & 1));
            }
            break;
        }
        const uint8_t myflag = threadIdx.x < 2 ? flag[(size_t)b * 2 + threadIdx.x] : (uint8_t)0;
        auto noload = [&](int) -> C2 { return cmk<C2>((T)0, (T)0); };
        if constexpr (Z3) {
            if constexpr (G % 16 == 0 || (sizeof(T) == 8 && N > 128)) {
                for (int q = g; q < M / 2; q += G) split3_pre<T, M, SUB>(fa, fb, tw3, tiles + tbase, q);
            } else {   // see k_zpass
                for (int idx = threadIdx.x; idx < 9 * (M / 2); idx += 9 * G) {
                    const int tj = idx / (M / 2), v = tj / 3, tq = tj - 3 * v;
                    const C2* const f0 = stage + (tq < 2 ? (v * 3 * 2 + tq) * KZP : (v * 3 + 2) * 2 * KZP);
                    split3_pre<T, M, SUB>(f0, f0 + (tq < 2 ? 2 * KZP : KZP), tw3, tiles + tj * LP, idx % (M / 2));
                }
            }
            __syncthreads();
            // every read of the staging buffer is done, the next batch may land
            if (threadIdx.x == 0 && more) issue(b + gridDim.x);
            const int sub = g / GM, gm = g % GM;
            if constexpr (PAD) {
                S3::template FFT<1, WS>::template run_tile<true>(tiles, tw, Pad16{tbase + sub * SUB}, gm, noload);
            } else {
                auto addr = [&](int r) { return tbase + zaddr(sub * M + r, 0, 0); };
                auto store = [&](int r, C2 v) { tiles[addr(r)] = v; };
                S3::template FFT<1, WS>::template run<true>(tiles, tw, addr, gm, noload, store);
            }
        } else {
            auto load = [&](int q) -> C2 {
                if (q < Kz) {
                    C2 a = fa[q], c = fb[q];
                    if (q == 0) { a.y = 0; c.y = 0; }
                    return cmk<C2>(a.x - c.y, a.y + c.x);          // A + i B
                }
                if (q > N - Kz) {
                    const C2 a = fa[N - q], c = fb[N - q];
                    return cmk<C2>(a.x + c.y, c.x - a.y);          // conj(A) + i conj(B)
                }
                return cmk<C2>((T)0, (T)0);
            };
            LineFFT<T, N, 1, WS>::template run_tile<false>(tiles, tw, Pad16{tbase}, g, load);
        }
        if (threadIdx.x < 2) sflag[threadIdx.x] = myflag;
        __syncthreads();
        if (!Z3 && threadIdx.x == 0 && more) issue(b + gridDim.x);
        // pointwise, both lines at one z per thread and round: the thread
        // alone reads and writes these slots
        for (int z = threadIdx.x; z < N; z += blockDim.x) {
            C2* const t = tiles + zpos(z);
            const uint32_t lid = 2u * (uint32_t)b, x = lid / NY, y0 = lid - x * NY;   // NY is even: one x-plane
            const C2 uz = t[2 * LP], wz = t[5 * LP], bz = t[8 * LP];
            T ub3[2], wb3[2];
#pragma unroll
            for (int ln = 0; ln < 2; ++ln) {
                const size_t po = (size_t)(lid + ln) * N + z;
                const T sx = us[po], sy = us[N3 + po], sz = us[2 * N3 + po];
                const T c = sflag[ln] ? chi[po] : (T)0;
                const C2 u = t[ln * LP], w = t[(3 + ln) * LP], nv = t[(6 + ln) * LP];
                const T u2 = ln ? uz.y : uz.x, w2 = ln ? wz.y : wz.x;
                const T n0 = nv.x * invn3, n1 = nv.y * invn3, n2 = (ln ? bz.y : bz.x) * invn3;
                const T rx = (T)(int)x * dx - (T)kp.x0[0], ry = (T)(int)(y0 + ln) * dx - (T)kp.x0[1],
                        rz = (T)z * dx - (T)kp.x0[2];
                const T ce = c * inv_eta, cf = fs * c;
                // the force and moment term uses dJ/dp = a + b x r, p = chi (u - us);
                // dJ/dchi is needed at every cell (also where chi = 0)
                const T gx = a0 + b1 * rz - b2 * ry;
                const T gy = a1 + b2 * rx - b0 * rz;
                const T gz = a2 + b0 * ry - b1 * rx;
                // ubar = w x nbar - c nbar + cf g; wbar = nbar x u
                t[ln * LP] = cmk<C2>(w.y * n2 - w2 * n1 - ce * n0 + cf * gx, w2 * n0 - w.x * n2 - ce * n1 + cf * gy);
                ub3[ln] = w.x * n1 - w.y * n0 - ce * n2 + cf * gz;
                t[(3 + ln) * LP] = cmk<C2>(n1 * u2 - n2 * u.y, n2 * u.x - n0 * u2);
                wb3[ln] = n0 * u.y - n1 * u.x;
                const T ex = u.x - sx, ey = u.y - sy, ez = u2 - sz;
                gchi[po] = -inv_eta * (n0 * ex + n1 * ey + n2 * ez) + fs * (gx * ex + gy * ey + gz * ez);
                gus[po] = ce * n0 - cf * gx;
                gus[N3 + po] = ce * n1 - cf * gy;
                gus[2 * N3 + po] = ce * n2 - cf * gz;
            }
            t[2 * LP] = cmk<C2>(ub3[0], ub3[1]);
            t[5 * LP] = cmk<C2>(wb3[0], wb3[1]);
        }
        __syncthreads();
        const bool active = vec < 2;
        if constexpr (Z3) {
            const int sub = g / GM, gm = g % GM;
            if constexpr (PAD) {
                S3::template FFT<-1, WS>::template run_tile_masked<true>(tiles, tw, Pad16{tbase + sub * SUB}, gm, noload,
                                                                        active);
            } else {
                auto addr = [&](int r) { return tbase + zaddr(sub * M + r, 0, 0); };
                auto store = [&](int r, C2 v) { if (active) tiles[addr(r)] = v; };
                S3::template FFT<-1, WS>::template run_masked<true>(tiles, tw, addr, gm, noload, store, active);
            }
        } else {
            LineFFT<T, N, -1, WS>::template run_tile_masked<true>(tiles, tw, Pad16{tbase}, g, noload, active);
        }
        __syncthreads();
        // unpack the two-for-one transforms: P = (Z_k + conj Z_{-k}) / 2 and
        // Q = (Z_k - conj Z_{-k}) / (2 i)
        auto P2 = [](C2 zk, C2 zm) { return cmk<C2>((T)0.5 * (zk.x + zm.x), (T)0.5 * (zk.y - zm.y)); };
        auto Q2 = [](C2 zk, C2 zm) { return cmk<C2>((T)0.5 * (zk.y + zm.y), (T)0.5 * (zm.x - zk.x)); };
        const int KH = Z3 ? M / 2 : Kz;   // items per tile
        for (int idx = threadIdx.x; idx < 6 * KH; idx += blockDim.x) {
            const int tj = idx / KH, k = idx - tj * KH, vf = tj / 3, tq = tj - 3 * vf;
            const C2* const t = tiles + tj * LP;
            // x and y of line tq, or z of both lines
            C2* const dP = B + (3 * vf + (tq < 2 ? 0 : 2)) * BS + ((size_t)b * 2 + (tq < 2 ? tq : 0)) * KZP;
            C2* const dQ = tq < 2 ? dP + BS : dP + KZP;
            if constexpr (Z3) {
                C2 zk, znk, zm, znm;
                split3_pair_out<T, M, SUB>(t, tw3, k, zk, znk, zm, znm);
                const int k2 = k == 0 ? M / 2 : M - k;
                dP[k] = P2(zk, znk);
                dQ[k] = Q2(zk, znk);
                dP[k2] = P2(zm, znm);
                dQ[k2] = Q2(zm, znm);
            } else {
                const int m = (N - k) % N;
                const C2 zk = t[k + (k >> 4)], zm = t[m + (m >> 4)];
                dP[k] = P2(zk, zm);
                dQ[k] = Q2(zk, zm);
            }
        }
        __syncthreads();
    }
}

}  // namespace ps
