// Fit, harmonic surface mapping and energy/forces (Sec. II.A-C).
//
//  fit_fp64          b from the monitoring potentials (periodic:
//                    b_i = Phi_in(x~_i) - Phi_in(x_i); grounded: b_i = -Phi_in(x_i))
//                    and A = M+ b (FP64 matrix-vector product per system).
//  surface_charges   at each integration direction u_j: Phi_out(Rs u_j) and
//                    sigma(Rs u_j) = (1/Rs) sum n A_nm B_nm(Rs u_j); the point
//                    images carry Q_sigma = w sigma/(4 pi) at Rs u_j and the
//                    dipole pair +-p/dr, p = w Phi_out/(4 pi), at (Rs -+ dr/2) u_j
//                    (Eqs. "green", "cd", "integrals" and the Fibonacci rule).
//  surface_pairs     potential and field of those images at every particle.
//  finalize          U = 1/2 sum q_i (Phi_in + Phi_out), F_i = q_i E_i.
#include <math.h>

#include "common.cuh"

namespace hsma {

namespace {

constexpr double kPi = 3.14159265358979323846;

// A = M+ b, a row per S of a block's eight warps (S = 8: one system's few rows
// over many SMs -- p = 10, K = 1500 has 120 rows, 15 blocks of eight and 47
// dependent rounds each before; S = 1: batches).  The S partial sums are added
// in warp order.
template <int S>
__global__ void __launch_bounds__(256) fit_fp64_kernel(const SysDesc *sys, int bc, int K, int ncols, int Nb,
                                                       const double *Mp, const double *phi_tgt, const int *mon_inv,
                                                       double *b_out, double *A)
{
    __shared__ double red[8];
    const SysDesc sd = sys[blockIdx.y];
    const double *ph = phi_tgt + sd.tgt_off + sd.n;  // monitoring targets
    const int drop = (bc == HSMA_BC_PERIODIC) ? 1 : 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * (8 / S) + warp / S;
    if (blockIdx.x == 0) {
        for (int i = threadIdx.x; i < K; i += blockDim.x)
            b_out[(long long)blockIdx.y * K + i] = rhs_at(ph, mon_inv, K, i, drop != 0);
        if (drop && threadIdx.x == 0) A[(long long)blockIdx.y * Nb] = 0.0;
    }
    double s = 0.0;
    if (c < ncols) {
        const double *row = Mp + (long long)c * K;
        for (int i = (warp % S) * 32 + lane; i < K; i += 32 * S) s += row[i] * rhs_at(ph, mon_inv, K, i, drop != 0);
    }
    s = warp_sum(s);
    if (S > 1) {
        if (lane == 0) red[warp] = s;
        __syncthreads();
        if (warp % S != 0) return;
        s = 0.0;
        for (int k = 0; k < S; ++k) s += red[warp + k];
    }
    if (lane == 0 && c < ncols) A[(long long)blockIdx.y * Nb + c + drop] = s;
}

__device__ __forceinline__ int degree_of(int k)
{
    int n = (int)sqrt((double)k);
    while (n * n > k) --n;
    while ((n + 1) * (n + 1) <= k) ++n;
    return n;
}

// Sigma and dipole images of kChargeDirs directions of a system per block, a
// warp per direction at a time; A and n A_nm staged once per block, so that an
// element takes two FP64 operations (FP64 issue bounds batches: 0.33 -> 0.18 ms
// for 32 systems at p = 10).  img: double2 (Q_sigma, p), or with f32 the same
// pairs as float2 for the FP32 surface sums, whose blocks then stage them
// without a conversion each.
constexpr int kChargeDirs = 16;
__global__ void __launch_bounds__(256) surface_charges_kernel(int ndir, int Nb, const double *Bq,
                                                              const double4_32a *dirs, const double *A, double Rs,
                                                              int f32, double2 *img)
{
    extern __shared__ double2 an[];  // (A_nm, n A_nm)
    const double *a = A + (long long)blockIdx.y * Nb;
    for (int k = threadIdx.x; k < Nb; k += blockDim.x) {
        const double v = a[k];
        an[k] = make_double2(v, degree_of(k) * v);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int hi = min(ndir, (int)(blockIdx.x + 1) * kChargeDirs);
    for (int d = blockIdx.x * kChargeDirs + (threadIdx.x >> 5); d < hi; d += 8) {
        const double *row = Bq + (long long)d * Nb;
        double phi = 0.0, sig = 0.0;
#pragma unroll 4
        for (int k = lane; k < Nb; k += 32) {
            const double v = row[k];
            const double2 c = an[k];
            phi = fma(v, c.x, phi);
            sig = fma(v, c.y, sig);
        }
        phi = warp_sum(phi);
        sig = warp_sum(sig);
        if (lane == 0) {
            const double w = dirs[d].w, q = w * sig / (Rs * 4.0 * kPi), p = w * phi / (4.0 * kPi);
            const long long o = (long long)blockIdx.y * ndir + d;
            if (f32)
                reinterpret_cast<float2 *>(img)[o] = make_float2((float)q, (float)p);
            else
                img[o] = make_double2(q, p);
        }
    }
}

// A block of kSurfThreads = kSurfSplit x kSurfGroup threads covers kSurfTB
// particles (kSurfT per thread); the kSurfSplit thread groups take every
// kSurfSplit-th direction of each staged tile (more warps per SM for the
// same work), and their partial sums are added in group order at the end.
constexpr int kSurfThreads = 256;
constexpr int kSurfSplit = 8;
constexpr int kSurfGroup = kSurfThreads / kSurfSplit;
constexpr int kSurfT = 2;
constexpr int kSurfTB = kSurfGroup * kSurfT;
constexpr int kSurfTile = 256;

__device__ __forceinline__ int find_sys_surf(const SysDesc *sys, int nsys, int item)
{
    int lo = 0, hi = nsys - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (sys[mid].surf_off <= item)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// FP32 form for thick layers.  For direction u with d = r - Rs u, h = dr/2,
// a = u.d:
//   sigma image:  Q/|d|, field Q d/|d|^3
//   dipole pair:  (p/dr)(1/A - 1/B) with A = |d + h u|, B = |d - h u|
//                 = -2 p a / (A B (A + B))                  (no cancellation)
//   its field:    (p/dr)((d + h u)/A^3 - (d - h u)/B^3)
//                 = p [ -2 a (A^2 + A B + B^2) / ((A + B) A^3 B^3) d
//                       + (u/2)(1/A^3 + 1/B^3) ]
//
// Each thread takes two directions of its group per step with packed FP32
// instructions (fma/add/mul.rn.f32x2 on the pair); the group's directions
// of a staged tile are stored pair-interleaved: sx = (u_x, u_x', u_y, u_y'),
// sy = (u_z, u_z', Q, Q'), sz = (-2 p, -2 p', p/2, p'/2).  Slots beyond the
// tile hold a direction with Q = p = 0, which contributes exactly zero.
constexpr int kSurfPairs = kSurfTile / kSurfSplit / 2;  // direction pairs per group per tile

__global__ void __launch_bounds__(kSurfThreads, 2) surface_pairs_fp32_kernel(
    const SysDesc *sys, int nsys, const float4 *src_hi, const float4 *src_lo, int ndir, const float4 *dirs,
    const float2 *img, float Rs, float h, double *phi_out, double *e_out)
{
    __shared__ float4 sx[kSurfSplit][kSurfPairs], sy[kSurfSplit][kSurfPairs], sz[kSurfSplit][kSurfPairs];
    __shared__ float2 red[kSurfSplit - 1][kSurfT][4][kSurfGroup];  // partial sums of groups 1..
    const int s = find_sys_surf(sys, nsys, blockIdx.x);
    const SysDesc sd = sys[s];
    const int blk = blockIdx.x - sd.surf_off;
    const int gl = threadIdx.x % kSurfGroup;  // particle lane
    const int grp = threadIdx.x / kSurfGroup;  // direction group (uniform per warp)
    float2 RX[kSurfT], RY[kSurfT], RZ[kSurfT];  // particle position, both lanes
    long long idx[kSurfT];
#pragma unroll
    for (int t = 0; t < kSurfT; ++t) {
        long long i = sd.sp_lo + (long long)blk * kSurfTB + t * kSurfGroup + gl;
        const bool ok = i < sd.sp_lo + sd.sp_n;
        idx[t] = ok ? i : -1;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (ok) {
            a = src_hi[sd.src_off + i];
            b = src_lo[sd.src_off + i];
        }
        const float rx = a.x + b.x, ry = a.y + b.y, rz = a.z + b.z;
        RX[t] = make_float2(rx, rx);
        RY[t] = make_float2(ry, ry);
        RZ[t] = make_float2(rz, rz);
    }
    const float2 NRS = make_float2(-Rs, -Rs), HH = make_float2(h * h, h * h);
    const float2 H2 = make_float2(2.f * h, 2.f * h), NH2 = make_float2(-2.f * h, -2.f * h);
    float2 phi[kSurfT], e[kSurfT][3];
#pragma unroll
    for (int t = 0; t < kSurfT; ++t) {
        phi[t] = make_float2(0.f, 0.f);
        e[t][0] = e[t][1] = e[t][2] = make_float2(0.f, 0.f);
    }
    const float2 *im = img + (long long)s * ndir;
    float *fx = reinterpret_cast<float *>(&sx[0][0]), *fy = reinterpret_cast<float *>(&sy[0][0]);
    float *fz = reinterpret_cast<float *>(&sz[0][0]);
    for (int d0 = 0; d0 < ndir; d0 += kSurfTile) {
        const int cnt = min(kSurfTile, ndir - d0);
        __syncthreads();
        for (int j = threadIdx.x; j < kSurfTile; j += kSurfThreads) {
            float ux = 1.f, uy = 0.f, uz = 0.f, Q = 0.f, pw = 0.f;
            if (j < cnt) {
                const float4 u = dirs[d0 + j];
                const float2 c = im[d0 + j];
                ux = u.x;
                uy = u.y;
                uz = u.z;
                Q = u.w > 0.f ? c.x : 0.f;
                pw = u.w > 0.f ? c.y : 0.f;
            }
            const int g = j % kSurfSplit, k = j / kSurfSplit, kp = k >> 1, ln = k & 1;
            const int base = (g * kSurfPairs + kp) * 4;
            fx[base + ln] = ux;
            fx[base + 2 + ln] = uy;
            fy[base + ln] = uz;
            fy[base + 2 + ln] = Q;
            fz[base + ln] = -2.f * pw;
            fz[base + 2 + ln] = 0.5f * pw;
        }
        __syncthreads();
        const int cg = cnt > grp ? (cnt - grp + kSurfSplit - 1) / kSurfSplit : 0;  // this group's directions
        const int npairs = (cg + 1) >> 1;
        float2 pa[kSurfT], ea[kSurfT][3];
#pragma unroll
        for (int t = 0; t < kSurfT; ++t) {
            pa[t] = make_float2(0.f, 0.f);
            ea[t][0] = ea[t][1] = ea[t][2] = make_float2(0.f, 0.f);
        }
#pragma unroll 2
        for (int kp = 0; kp < npairs; ++kp) {
            const float4 X = sx[grp][kp], Y = sy[grp][kp], Z = sz[grp][kp];
            const float2 ux = make_float2(X.x, X.y), uy = make_float2(X.z, X.w);
            const float2 uz = make_float2(Y.x, Y.y), Q = make_float2(Y.z, Y.w);
            const float2 np2 = make_float2(Z.x, Z.y), hp = make_float2(Z.z, Z.w);
#pragma unroll
            for (int t = 0; t < kSurfT; ++t) {
                const float2 dx = __ffma2_rn(NRS, ux, RX[t]);
                const float2 dy = __ffma2_rn(NRS, uy, RY[t]);
                const float2 dz = __ffma2_rn(NRS, uz, RZ[t]);
                const float2 dd = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                const float2 ad = __ffma2_rn(ux, dx, __ffma2_rn(uy, dy, __fmul2_rn(uz, dz)));
                const float2 base = __fadd2_rn(dd, HH);
                const float2 A2 = __ffma2_rn(H2, ad, base);
                const float2 B2 = __ffma2_rn(NH2, ad, base);
                const float2 ri = make_float2(rsqrt_sfu(dd.x), rsqrt_sfu(dd.y));
                const float2 Ai = make_float2(rsqrt_sfu(A2.x), rsqrt_sfu(A2.y));
                const float2 Bi = make_float2(rsqrt_sfu(B2.x), rsqrt_sfu(B2.y));
                const float2 Aa = __fmul2_rn(A2, Ai), Bb = __fmul2_rn(B2, Bi);
                const float2 sab = __fadd2_rn(Aa, Bb);
                const float2 inv = make_float2(__fdividef(1.f, sab.x), __fdividef(1.f, sab.y));
                const float2 qs = __fmul2_rn(Q, ri);
                const float2 m1 = __fmul2_rn(np2, ad);                                   // -2 p a
                const float2 dip = __fmul2_rn(__fmul2_rn(m1, __fmul2_rn(Ai, Bi)), inv);  // dipole potential
                pa[t] = __fadd2_rn(pa[t], __fadd2_rn(qs, dip));
                const float2 ri3 = __fmul2_rn(__fmul2_rn(ri, ri), ri);
                const float2 Ai3 = __fmul2_rn(__fmul2_rn(Ai, Ai), Ai);
                const float2 Bi3 = __fmul2_rn(__fmul2_rn(Bi, Bi), Bi);
                const float2 S = __fadd2_rn(__ffma2_rn(Aa, Bb, A2), B2);  // A^2 + A B + B^2
                const float2 cd = __fadd2_rn(
                    __fmul2_rn(Q, ri3), __fmul2_rn(__fmul2_rn(__fmul2_rn(__fmul2_rn(m1, S), inv), Ai3), Bi3));
                const float2 cu = __fmul2_rn(hp, __fadd2_rn(Ai3, Bi3));
                ea[t][0] = __fadd2_rn(ea[t][0], __ffma2_rn(cd, dx, __fmul2_rn(cu, ux)));
                ea[t][1] = __fadd2_rn(ea[t][1], __ffma2_rn(cd, dy, __fmul2_rn(cu, uy)));
                ea[t][2] = __fadd2_rn(ea[t][2], __ffma2_rn(cd, dz, __fmul2_rn(cu, uz)));
            }
        }
#pragma unroll
        for (int t = 0; t < kSurfT; ++t) {
            phi[t] = df_add(phi[t], pa[t].x + pa[t].y);
            e[t][0] = df_add(e[t][0], ea[t][0].x + ea[t][0].y);
            e[t][1] = df_add(e[t][1], ea[t][1].x + ea[t][1].y);
            e[t][2] = df_add(e[t][2], ea[t][2].x + ea[t][2].y);
        }
    }
    // add the groups' partial sums in group order
    if (grp > 0) {
#pragma unroll
        for (int t = 0; t < kSurfT; ++t) {
            red[grp - 1][t][0][gl] = phi[t];
            red[grp - 1][t][1][gl] = e[t][0];
            red[grp - 1][t][2][gl] = e[t][1];
            red[grp - 1][t][3][gl] = e[t][2];
        }
    }
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int t = 0; t < kSurfT; ++t) {
#pragma unroll
        for (int g2 = 0; g2 < kSurfSplit - 1; ++g2) {
            phi[t] = df_add_df(phi[t], red[g2][t][0][gl]);
            e[t][0] = df_add_df(e[t][0], red[g2][t][1][gl]);
            e[t][1] = df_add_df(e[t][1], red[g2][t][2][gl]);
            e[t][2] = df_add_df(e[t][2], red[g2][t][3][gl]);
        }
        if (idx[t] < 0) continue;
        long long o = sd.part_off + idx[t];
        phi_out[o] = (double)phi[t].x + (double)phi[t].y;
        e_out[3 * o] = (double)e[t][0].x + (double)e[t][0].y;
        e_out[3 * o + 1] = (double)e[t][1].x + (double)e[t][1].y;
        e_out[3 * o + 2] = (double)e[t][2].x + (double)e[t][2].y;
    }
}

// FP32 form for thin layers: the dipole pair as its Legendre series (see the
// FP64 form below), with d, a = -u.d and rho = |d|:
//   potential  Q/rho + m (1 + k0),                     m = p a/rho^3
//   field      (Q/rho^3 + (3 m/rho^2)(1 + k2)) d + (p/rho^3)(1 + k1) u
//   k0 = s (5 q^2 - 3), k1 = s (15 q^2 - 3), k2 = s (35 q^2 - 15)/3,
//   s = h^2/(2 rho^2), q = a/rho;
// H2 = false leaves the k's out where they are below the FP32 rounding
// (12 s < 6e-9), and the next terms, (h/rho)^4, are below it up to h = 5e-3 rho.
// 24 (with the k's 36) FP32 lane operations and one SFU result per direction
// and particle against about 50 and four of the literal form above.
//
// A block of 256 threads is G direction groups of 256/G lanes with T particles
// each; the directions of a staged tile go round the groups, two per packed
// instruction.  G = 8, T = 2 (64 particles a block) for large systems;
// G = 32, T = 1 (8 particles) where that leaves SMs without a block.  The
// FP32 directions come from the plan and the images in FP32 from
// surface_charges: staging converted seven FP64 values per direction and
// block before, at two per SM and clock.
// Measured: N = 100000, 3196 directions 0.533 -> 0.293 ms; N = 4000 0.066 ->
// 0.029; N = 500, 1976 directions 0.043 -> 0.014; with the k's, grounded
// N = 20000 0.102 -> 0.078; 32 boxes of 500..50000 0.731 -> 0.397.
template <int G, int T, bool H2>
__global__ void __launch_bounds__(256) surface_dipole_fp32_kernel(const SysDesc *sys, int nsys, const float4 *src_hi,
                                                                  const float4 *src_lo, int ndir, const float4 *dirs,
                                                                  const float2 *img, float Rs, float hh,
                                                                  double *phi_out, double *e_out)
{
    constexpr int L = 256 / G, kPairs = kSurfTile / 2;
    // direction pairs: (ux, ux', uy, uy'), (uz, uz', Q, Q'), (p, p')
    __shared__ float4 sx[kPairs], sy[kPairs];
    __shared__ float2 sz[kPairs];
    __shared__ float2 red[G - 1][T][4][L];  // partial sums of groups 1..
    const int s = find_sys_surf(sys, nsys, blockIdx.x);
    const SysDesc sd = sys[s];
    const int gl = threadIdx.x % L, grp = threadIdx.x / L;
    const long long hi = sd.sp_lo + sd.sp_n;
    const long long i0 = sd.sp_lo + (long long)(blockIdx.x - sd.surf_off) * kSurfTB + (long long)blockIdx.y * L * T;
    if (i0 >= hi) return;
    float2 RX[T], RY[T], RZ[T];  // particle position, both lanes
    long long idx[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        const long long i = i0 + t * L + gl;
        idx[t] = i < hi ? i : -1;
        const float4 a = src_hi[sd.src_off + min(i, hi - 1)], b = src_lo[sd.src_off + min(i, hi - 1)];
        const float rx = a.x + b.x, ry = a.y + b.y, rz = a.z + b.z;
        RX[t] = make_float2(rx, rx);
        RY[t] = make_float2(ry, ry);
        RZ[t] = make_float2(rz, rz);
    }
    const float2 NRS = make_float2(-Rs, -Rs), M1 = make_float2(-1.f, -1.f), C3 = make_float2(3.f, 3.f);
    float2 phi[T], e[T][3];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        phi[t] = make_float2(0.f, 0.f);
        e[t][0] = e[t][1] = e[t][2] = make_float2(0.f, 0.f);
    }
    const float2 *im = img + (long long)s * ndir;
    for (int d0 = 0; d0 < ndir; d0 += kSurfTile) {
        __syncthreads();
        for (int j = threadIdx.x; j < kPairs; j += 256) {
            // beyond the last direction: one without images
            const int a = d0 + 2 * j, b = a + 1;
            const float4 u = a < ndir ? dirs[a] : make_float4(1.f, 0.f, 0.f, 0.f);
            const float4 v = b < ndir ? dirs[b] : make_float4(1.f, 0.f, 0.f, 0.f);
            const float2 c = a < ndir ? im[a] : make_float2(0.f, 0.f), f = b < ndir ? im[b] : make_float2(0.f, 0.f);
            sx[j] = make_float4(u.x, v.x, u.y, v.y);
            sy[j] = make_float4(u.z, v.z, c.x, f.x);
            sz[j] = make_float2(c.y, f.y);
        }
        __syncthreads();
        const int npairs = min(kPairs, (ndir - d0 + 1) >> 1);
        float2 pa[T], ea[T][3];
#pragma unroll
        for (int t = 0; t < T; ++t) {
            pa[t] = make_float2(0.f, 0.f);
            ea[t][0] = ea[t][1] = ea[t][2] = make_float2(0.f, 0.f);
        }
#pragma unroll 2
        for (int kp = grp; kp < npairs; kp += G) {
            const float4 X = sx[kp], Y = sy[kp];
            const float2 p = sz[kp];
            const float2 ux = make_float2(X.x, X.y), uy = make_float2(X.z, X.w);
            const float2 uz = make_float2(Y.x, Y.y), Q = make_float2(Y.z, Y.w);
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const float2 dx = __ffma2_rn(NRS, ux, RX[t]);
                const float2 dy = __ffma2_rn(NRS, uy, RY[t]);
                const float2 dz = __ffma2_rn(NRS, uz, RZ[t]);
                const float2 dd = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                const float2 na = __ffma2_rn(ux, dx, __ffma2_rn(uy, dy, __fmul2_rn(uz, dz)));  // -a
                const float2 ri = make_float2(rsqrt_sfu(dd.x), rsqrt_sfu(dd.y));
                const float2 ri2 = __fmul2_rn(ri, ri), ri3 = __fmul2_rn(ri2, ri);
                float2 w = __fmul2_rn(p, ri3);
                float2 m = __fmul2_rn(__fmul2_rn(w, na), M1);
                float2 m3 = __fmul2_rn(m, ri2);
                if (H2) {
                    const float2 qq = __fmul2_rn(__fmul2_rn(na, na), ri2);
                    const float2 sc = __fmul2_rn(make_float2(hh, hh), ri2);
                    const float2 k0 = __ffma2_rn(make_float2(5.f, 5.f), qq, make_float2(-3.f, -3.f));
                    const float2 k1 = __ffma2_rn(make_float2(15.f, 15.f), qq, make_float2(-3.f, -3.f));
                    const float2 k2 = __ffma2_rn(make_float2(35.f / 3.f, 35.f / 3.f), qq, make_float2(-5.f, -5.f));
                    m = __ffma2_rn(m, __fmul2_rn(sc, k0), m);
                    w = __ffma2_rn(w, __fmul2_rn(sc, k1), w);
                    m3 = __ffma2_rn(m3, __fmul2_rn(sc, k2), m3);
                }
                pa[t] = __fadd2_rn(__ffma2_rn(Q, ri, pa[t]), m);
                const float2 cd = __ffma2_rn(C3, m3, __fmul2_rn(Q, ri3));
                ea[t][0] = __ffma2_rn(cd, dx, __ffma2_rn(w, ux, ea[t][0]));
                ea[t][1] = __ffma2_rn(cd, dy, __ffma2_rn(w, uy, ea[t][1]));
                ea[t][2] = __ffma2_rn(cd, dz, __ffma2_rn(w, uz, ea[t][2]));
            }
        }
#pragma unroll
        for (int t = 0; t < T; ++t) {
            phi[t] = df_add(phi[t], pa[t].x + pa[t].y);
            e[t][0] = df_add(e[t][0], ea[t][0].x + ea[t][0].y);
            e[t][1] = df_add(e[t][1], ea[t][1].x + ea[t][1].y);
            e[t][2] = df_add(e[t][2], ea[t][2].x + ea[t][2].y);
        }
    }
    // add the groups' partial sums in group order
    if (grp > 0) {
#pragma unroll
        for (int t = 0; t < T; ++t) {
            red[grp - 1][t][0][gl] = phi[t];
            red[grp - 1][t][1][gl] = e[t][0];
            red[grp - 1][t][2][gl] = e[t][1];
            red[grp - 1][t][3][gl] = e[t][2];
        }
    }
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int t = 0; t < T; ++t) {
#pragma unroll 7
        for (int g2 = 0; g2 < G - 1; ++g2) {
            phi[t] = df_add_df(phi[t], red[g2][t][0][gl]);
            e[t][0] = df_add_df(e[t][0], red[g2][t][1][gl]);
            e[t][1] = df_add_df(e[t][1], red[g2][t][2][gl]);
            e[t][2] = df_add_df(e[t][2], red[g2][t][3][gl]);
        }
        if (idx[t] < 0) continue;
        const long long o = sd.part_off + idx[t];
        phi_out[o] = (double)phi[t].x + (double)phi[t].y;
        e_out[3 * o] = (double)e[t][0].x + (double)e[t][0].y;
        e_out[3 * o + 1] = (double)e[t][1].x + (double)e[t][1].y;
        e_out[3 * o + 2] = (double)e[t][2].x + (double)e[t][2].y;
    }
}

// FP64 form for thick dipole layers: the three point images of each direction
// summed literally; one particle per thread, kSurfTB per block (the FP32
// kernel's block size).
constexpr int kSurf64Threads = kSurfTB;
__global__ void __launch_bounds__(kSurf64Threads) surface_pairs_fp64_kernel(
    const SysDesc *sys, int nsys, const double4_32a *src64, int ndir, const double4_32a *dirs, const double2 *img,
    double Rs, double dr, double *phi_out, double *e_out)
{
    __shared__ double4_32a su[kSurfTile];
    __shared__ double sp[kSurfTile];
    const int s = find_sys_surf(sys, nsys, blockIdx.x);
    const SysDesc sd = sys[s];
    const int blk = blockIdx.x - sd.surf_off;
    constexpr int T = 1;
    double r[T][3];
    long long idx[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        long long i = sd.sp_lo + (long long)blk * kSurfTB + t * kSurf64Threads + threadIdx.x;
        const bool ok = i < sd.sp_lo + sd.sp_n;
        idx[t] = ok ? i : -1;
        double4_32a a = make_double4_32a(0, 0, 0, 0);
        if (ok) a = src64[sd.src_off + i];
        r[t][0] = a.x;
        r[t][1] = a.y;
        r[t][2] = a.z;
    }
    double phi[T], e[T][3];
#pragma unroll
    for (int t = 0; t < T; ++t) phi[t] = e[t][0] = e[t][1] = e[t][2] = 0.0;
    const double2 *im = img + (long long)s * ndir;
    const double Rin = Rs - 0.5 * dr, Rout = Rs + 0.5 * dr;
    for (int d0 = 0; d0 < ndir; d0 += kSurfTile) {
        int cnt = min(kSurfTile, ndir - d0);
        __syncthreads();
        for (int j = threadIdx.x; j < cnt; j += kSurf64Threads) {
            double4_32a u = dirs[d0 + j];
            double2 c = im[d0 + j];
            su[j] = make_double4_32a(u.x, u.y, u.z, c.x);
            sp[j] = c.y / dr;
        }
        __syncthreads();
        for (int j = 0; j < cnt; ++j) {
            const double4_32a u = su[j];
            const double pd = sp[j];
            const double R3[3] = {Rs, Rin, Rout};
            const double Q3[3] = {u.w, pd, -pd};
#pragma unroll
            for (int t = 0; t < T; ++t) {
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    double dx = r[t][0] - R3[m] * u.x;
                    double dy = r[t][1] - R3[m] * u.y;
                    double dz = r[t][2] - R3[m] * u.z;
                    double ri = rsqrt(dx * dx + dy * dy + dz * dz);
                    double qr = Q3[m] * ri;
                    phi[t] += qr;
                    double qr3 = qr * ri * ri;
                    e[t][0] += qr3 * dx;
                    e[t][1] += qr3 * dy;
                    e[t][2] += qr3 * dz;
                }
            }
        }
    }
#pragma unroll
    for (int t = 0; t < T; ++t) {
        if (idx[t] < 0) continue;
        long long o = sd.part_off + idx[t];
        phi_out[o] = phi[t];
        e_out[3 * o] = e[t][0];
        e_out[3 * o + 1] = e[t][1];
        e_out[3 * o + 2] = e[t][2];
    }
}

// FP64 form for thin dipole layers.  With d = r - Rs u, a = -u.d (> 0: the
// particle is inside the sphere) and rho = |d|, the pair (p/dr)(1/A - 1/B) of
// the literal form is the odd part of the Legendre series of 1/|d + s u| at
// s = dr/2 = h,
//   p [ a/rho^3 + h^2 P3(a/rho)/rho^4 + O(h^4/rho^6) ]:
// a point dipole, and an h^2 term 1e-10 of it (dr = 1e-5 Rs) that FP32 holds
// to the last FP64 bit.  The series leaves out (h/rho)^4 of the dipole, where
// the literal difference of two 1/dr terms rounds at 2^-53 rho/h of it, so it
// is the more accurate form while h <= 6.4e-4 rho (launch_surface_pairs).  rho^2
// and E below are rounded by up to 2^-53 (Rs/rho)^2, also less than that: at the
// corners of boxes 1% to 30% inside their sphere, 540 to 2e5 directions, the
// field's rms error is 0.001 to 0.94 times the literal form's.
//
// FP64 issue bounds both forms: 26 FP64 operations here per direction and
// particle against 57 of the literal form.  A warp takes one particle and
// every 32nd direction, so that small systems fill the chip as well (a thread
// per particle left 16 blocks at N = 1000) and large ones leave a short tail:
// two and four particles per warp, which share the loads, took 3% and 12%
// longer.  N = 9999, 3196 directions: 6.35 -> 1.56 ms (79% of the FP64 rate);
// N = 1000, 756: 1.38 -> 0.057 ms; grounded N = 3001, 1976: 3.60 -> 0.30 ms.
//
// f32_bits: v 2^-e in FP32 (truncated; 0 below 2^-126) by integer operations:
// a conversion would take a slot of the FP64 pipe.
__device__ __forceinline__ float f32_bits(double v, int e)
{
    const int hi = __double2hiint(v), m = (hi & 0x7fffffff) - ((896 + e) << 20);
    const int b = m > 0 ? (m << 3) | (int)((unsigned)__double2loint(v) >> 29) : 0;
    return __int_as_float((hi & (int)0x80000000u) | b);
}

__global__ void __launch_bounds__(128) surface_dipole_fp64_kernel(
    const SysDesc *sys, int nsys, const double4_32a *src64, int ndir, const double4_32a *dirs, const double2 *img,
    double Rs, double dr, double *phi_out, double *e_out)
{
    const int s = find_sys_surf(sys, nsys, blockIdx.x);
    const SysDesc sd = sys[s];
    const int lane = threadIdx.x & 31;
    const long long i = sd.sp_lo + (long long)(blockIdx.x - sd.surf_off) * kSurfTB + blockIdx.y * 4 +
                        (threadIdx.x >> 5);  // this warp's particle
    if (i >= sd.sp_lo + sd.sp_n) return;
    // the image dipoles' largest exponent, so that FP32 holds them whatever
    // the units: the h^2 term runs in units of Rs and 2^pe
    const double2 *im = img + (long long)s * ndir;
    int pe = 0;
    for (int j = lane; j < ndir; j += 32) pe = max(pe, (__double2hiint(im[j].y) & 0x7fffffff) >> 20);
    pe = __reduce_max_sync(0xffffffffu, pe);
    const double4_32a r = src64[sd.src_off + i];
    const float rx = (float)(r.x / Rs), ry = (float)(r.y / Rs), rz = (float)(r.z / Rs);
    const float h2 = (float)(0.25 * (dr / Rs) * (dr / Rs));
    const double c2 = fma(r.x, r.x, fma(r.y, r.y, fma(r.z, r.z, Rs * Rs)));
    // E = r S + K: the coefficient of d summed once, the rest per component
    double phi = 0.0, S = 0.0, Kx = 0.0, Ky = 0.0, Kz = 0.0;
    float pf = 0.f, ex = 0.f, ey = 0.f, ez = 0.f;
    for (int j = lane; j < ndir; j += 32) {
        const double4_32a u = dirs[j];
        const double2 c = im[j];
        const double ur = fma(u.x, r.x, fma(u.y, r.y, u.z * r.z));
        const double a = Rs - ur;
        const double ri = rsqrt(fma(-2.0 * Rs, ur, c2));
        const double ri2 = ri * ri, ri3 = ri2 * ri;
        const double w = c.y * ri3, m = w * a;
        phi = fma(c.x, ri, phi) + m;
        const double cd = fma(3.0 * m, ri2, c.x * ri3);
        const double k = fma(-Rs, cd, w);
        S += cd;
        Kx = fma(k, u.x, Kx);
        Ky = fma(k, u.y, Ky);
        Kz = fma(k, u.z, Kz);
        // h^2 term: p h^2 rho^-4 (5 q^3 - 3 q)/2 with q = a/rho, and minus its gradient
        const float ux = f32_bits(u.x, 0), uy = f32_bits(u.y, 0), uz = f32_bits(u.z, 0);
        const float dx = rx - ux, dy = ry - uy, dz = rz - uz;
        const float fi = rsqrt_sfu(fmaf(dx, dx, fmaf(dy, dy, dz * dz))), fi2 = fi * fi;
        const float q = -fmaf(ux, dx, fmaf(uy, dy, uz * dz)) * fi, qq = q * q;
        const float g4 = 0.5f * h2 * f32_bits(c.y, pe - 1023) * fi2 * fi2;
        pf = fmaf(g4 * q, fmaf(5.f, qq, -3.f), pf);
        const float cu = g4 * fi * fmaf(15.f, qq, -3.f), cv = g4 * fi2 * q * fmaf(35.f, qq, -15.f);
        ex = fmaf(cu, ux, fmaf(cv, dx, ex));
        ey = fmaf(cu, uy, fmaf(cv, dy, ey));
        ez = fmaf(cu, uz, fmaf(cv, dz, ez));
    }
    const double us = pe > 0 ? scalbn(1.0 / (Rs * Rs), pe - 1023) : 0.0, ue = us / Rs;
    phi = warp_sum(fma((double)pf, us, phi));
    S = warp_sum(S);
    Kx = warp_sum(fma((double)ex, ue, Kx));
    Ky = warp_sum(fma((double)ey, ue, Ky));
    Kz = warp_sum(fma((double)ez, ue, Kz));
    if (lane == 0) {
        const long long o = sd.part_off + i;
        phi_out[o] = phi;
        e_out[3 * o] = fma(S, r.x, Kx);
        e_out[3 * o + 1] = fma(S, r.y, Ky);
        e_out[3 * o + 2] = fma(S, r.z, Kz);
    }
}

// Forces, potentials and per-block energy partials of the particles a call
// owns: the sorted range [sp_lo, sp_lo + sp_n) of each system (all of it,
// except for a part of a target-sharded step).  Target i of a system is its
// i-th particle in spatial order; perm maps it back to the caller's index.
// Block b of system s covers particles [sp_lo + b kFinal, sp_lo + (b + 1) kFinal).
// owned_idx == nullptr: outputs at the caller's indices; otherwise (one
// system) output j is particle sp_lo + j and owned_idx[j] its caller index.
constexpr int kFinalThreads = 256;
constexpr int kFinal = 256;  // one particle per thread: 2048 left one or two blocks to systems of a few thousand

// The block that finishes last in its system (status[nsys + s] counts them)
// adds the partials -- a warp, each lane every 32nd in order, then a fixed
// tree, so the sum does not depend on which block it is -- and packs what the
// host reads into one record.
__global__ void __launch_bounds__(kFinalThreads) finalize_kernel(const SysDesc *sys, const int *perm, const double *q,
                                                                 const double *phi_tgt, const double *e_part,
                                                                 const double *phi_out, const double *e_out,
                                                                 double *forces, double *pot, long long *owned_idx,
                                                                 double *upart, int nb_max, double *energy,
                                                                 const long long *ns, int *status,
                                                                 StepResult *result)
{
    __shared__ double red[32];
    __shared__ int s_last;
    const int s = blockIdx.y;
    const SysDesc sd = sys[s];
    const int nb = max(1, (int)((sd.sp_n + kFinal - 1) / kFinal));
    if ((int)blockIdx.x >= nb) return;
    const long long i0 = sd.sp_lo + (long long)blockIdx.x * kFinal;
    const long long i1 = sd.sp_lo + sd.sp_n;
    double u = 0.0;
    bool bad = false;
    for (long long i = i0 + threadIdx.x; i < i1 && i < i0 + kFinal; i += blockDim.x) {
        long long t = sd.tgt_off + i, so = sd.part_off + i;
        const long long ci = sd.part_off + perm[so];  // caller's index
        double qi = q[ci];
        long long o = ci;
        if (owned_idx) {
            o = i - sd.sp_lo;
            owned_idx[o] = perm[so];
        }
        double ph = phi_tgt[t] + phi_out[so];
        double ex = e_part[3 * t] + e_out[3 * so];
        double ey = e_part[3 * t + 1] + e_out[3 * so + 1];
        double ez = e_part[3 * t + 2] + e_out[3 * so + 2];
        if (!isfinite(ph) || !isfinite(ex) || !isfinite(ey) || !isfinite(ez)) bad = true;
        if (forces) {
            forces[3 * o] = qi * ex;
            forces[3 * o + 1] = qi * ey;
            forces[3 * o + 2] = qi * ez;
        }
        if (pot) pot[o] = ph;
        u += qi * ph;
    }
    if (bad) atomicOr(&status[s], ST_COINCIDENT);
    u = block_sum(u, red);
    double *up = upart + (long long)s * nb_max;
    if (threadIdx.x == 0) {
        up[blockIdx.x] = u;
        __threadfence();
        s_last = atomicAdd(&status[gridDim.y + s], 1) == nb - 1;
    }
    __syncthreads();
    if (!s_last || threadIdx.x >= 32) return;
    __threadfence();
    u = 0.0;
    for (int b = threadIdx.x; b < nb; b += 32) u += __ldcg(up + b);
    u = warp_sum(u);
    if (threadIdx.x != 0) return;
    energy[s] = 0.5 * u;
    const int st = atomicOr(&status[s], isfinite(u) ? 0 : ST_COINCIDENT) | (isfinite(u) ? 0 : ST_COINCIDENT);
    result[s] = StepResult{0.5 * u, ns[s], st, 0};
}

}  // namespace

int launch_fit_fp64(const SysDesc *sys, int nsys, int bc, int K, int ncols, int Nb, const double *Mp,
                    const double *phi_tgt, const int *mon_inv, double *b_out, double *A, int num_sms, cudaStream_t st)
{
    if ((long long)ncols * nsys <= 8LL * num_sms)  // a block per row, at most eight per SM: all resident at once
        fit_fp64_kernel<8><<<dim3(ncols, nsys), 256, 0, st>>>(sys, bc, K, ncols, Nb, Mp, phi_tgt, mon_inv, b_out, A);
    else
        fit_fp64_kernel<1><<<dim3((ncols + 7) / 8, nsys), 256, 0, st>>>(sys, bc, K, ncols, Nb, Mp, phi_tgt, mon_inv,
                                                                       b_out, A);
    HSMA_LAUNCHED();
    HSMA_CUDA_TRY(cudaGetLastError());
    return HSMA_OK;
}

int launch_surface_charges(int nsys, int ndir, int Nb, const double *Bq, const double4_32a *dirs, const double *A,
                           double Rs, bool f32, double2 *img, cudaStream_t st)
{
    dim3 grid((ndir + kChargeDirs - 1) / kChargeDirs, nsys);
    surface_charges_kernel<<<grid, 256, Nb * sizeof(double2), st>>>(ndir, Nb, Bq, dirs, A, Rs, f32 ? 1 : 0, img);
    HSMA_LAUNCHED();
    HSMA_CUDA_TRY(cudaGetLastError());
    return HSMA_OK;
}

int surface_targets_per_block() { return kSurfTB; }

int launch_surface_pairs(const SysDesc *sys, int nsys, int total_items, const float4 *src_hi, const float4 *src_lo,
                         const double4_32a *src64, int ndir, const double4_32a *dirs, const float4 *dirs32,
                         const double2 *img, double Rs, double r_max, double dr, int precision, double *phi_out,
                         double *e_out, int num_sms, cudaStream_t st)
{
    if (total_items <= 0) return HSMA_OK;
    const double h = 0.5 * dr, rho = Rs - r_max;  // rho: a lower bound
    const float2 *img32 = reinterpret_cast<const float2 *>(img);
    if (precision == HSMA_FP64 && h <= 6.4e-4 * rho) {
        surface_dipole_fp64_kernel<<<dim3(total_items, kSurfTB / 4), 128, 0, st>>>(sys, nsys, src64, ndir, dirs, img,
                                                                                  Rs, dr, phi_out, e_out);
    } else if (precision == HSMA_FP64) {
        surface_pairs_fp64_kernel<<<total_items, kSurf64Threads, 0, st>>>(sys, nsys, src64, ndir, dirs, img, Rs, dr,
                                                                         phi_out, e_out);
    } else if (h <= 5e-3 * rho) {
        auto launch = [&](auto kernel, int particles) {
            kernel<<<dim3(total_items, kSurfTB / particles), 256, 0, st>>>(sys, nsys, src_hi, src_lo, ndir, dirs32,
                                                                          img32, (float)Rs, (float)(0.5 * h * h),
                                                                          phi_out, e_out);
        };
        const bool h2 = h > 3e-5 * rho;
        // blocks of 64 particles from the size where they are two per SM
        if (total_items >= 2 * num_sms)
            launch(h2 ? surface_dipole_fp32_kernel<8, 2, true> : surface_dipole_fp32_kernel<8, 2, false>, 64);
        else
            launch(h2 ? surface_dipole_fp32_kernel<32, 1, true> : surface_dipole_fp32_kernel<32, 1, false>, 8);
    } else {
        surface_pairs_fp32_kernel<<<total_items, kSurfThreads, 0, st>>>(sys, nsys, src_hi, src_lo, ndir, dirs32, img32,
                                                                       (float)Rs, (float)h, phi_out, e_out);
    }
    HSMA_LAUNCHED();
    HSMA_CUDA_TRY(cudaGetLastError());
    return HSMA_OK;
}

__global__ void directions_fp32_kernel(int n, const double4_32a *dirs, float4 *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double4_32a u = dirs[i];
    out[i] = make_float4((float)u.x, (float)u.y, (float)u.z, u.w > 0.0 ? 1.f : 0.f);
}

int launch_directions_fp32(int n, const double4_32a *dirs, float4 *out, cudaStream_t st)
{
    directions_fp32_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, dirs, out);
    HSMA_LAUNCHED();
    HSMA_CUDA_TRY(cudaGetLastError());
    return HSMA_OK;
}

int finalize_blocks(long long max_n) { return (int)((max_n + kFinal - 1) / kFinal); }

int launch_finalize(const SysDesc *sys, int nsys, long long max_n, const int *perm, const double *q,
                    const double *phi_tgt, const double *e_part, const double *phi_out, const double *e_out,
                    double *forces, double *pot, long long *owned_idx, double *upart, double *energy,
                    const long long *ns, int *status, StepResult *result, cudaStream_t st)
{
    const int nb_max = finalize_blocks(max_n);
    finalize_kernel<<<dim3(nb_max, nsys), kFinalThreads, 0, st>>>(sys, perm, q, phi_tgt, e_part, phi_out, e_out,
                                                                  forces, pot, owned_idx, upart, nb_max, energy, ns,
                                                                  status, result);
    HSMA_LAUNCHED();
    HSMA_CUDA_TRY(cudaGetLastError());
    return HSMA_OK;
}

int load_surface_kernels()
{
    return load_kernels(fit_fp64_kernel<8>, fit_fp64_kernel<1>, surface_charges_kernel, surface_pairs_fp32_kernel,
                        surface_pairs_fp64_kernel, surface_dipole_fp64_kernel, surface_dipole_fp32_kernel<8, 2, true>,
                        surface_dipole_fp32_kernel<8, 2, false>, surface_dipole_fp32_kernel<32, 1, true>,
                        surface_dipole_fp32_kernel<32, 1, false>, finalize_kernel);
}

}  // namespace hsma

namespace hsma {

namespace {

// Direct evaluation of the far field at the particles: Phi_out(r) =
// sum_k A_k B_k(r) (Eq. "harmonic") and E_out = -grad Phi_out, in FP64.  The
// basis is the orthonormal real solid harmonics of basis_kernel:
//   B = norm_k * Pi_n^m(z, r2) * Re/Im (x + i y)^m   (coordinates / Rs),
// with Pi from its three-term recurrence; the recurrence is differentiated
// alongside for dPi/dz and dPi/d(r2), so that
//   grad B = norm_k [ Pi grad(C_m|S_m) + (C_m|S_m)(dPi/dz e_z + 2 dPi/d(r2) r) ],
//   d/dx (C_m + i S_m) = m (C_{m-1} + i S_{m-1}),
//   d/dy (C_m + i S_m) = i m (C_{m-1} + i S_{m-1}).
__global__ void series_field_kernel(const SysDesc *sys, int nsys, int P, double inv_rs, const double *norm,
                                    const double *A, const float4 *src_hi, const float4 *src_lo,
                                    const double4_32a *src64, double *phi_out, double *e_out)
{
    const int s = blockIdx.y;
    const SysDesc sd = sys[s];
    const long long i = sd.sp_lo + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= sd.sp_lo + sd.sp_n) return;
    double x, y, z;
    if (src64) {
        double4_32a p = src64[sd.src_off + i];
        x = p.x; y = p.y; z = p.z;
    } else {
        float4 h = src_hi[sd.src_off + i], l = src_lo[sd.src_off + i];
        x = (double)h.x + (double)l.x;
        y = (double)h.y + (double)l.y;
        z = (double)h.z + (double)l.z;
    }
    x *= inv_rs; y *= inv_rs; z *= inv_rs;
    const double r2 = x * x + y * y + z * z;
    const int Nb = (P + 1) * (P + 1);
    const double *a = A + (long long)s * Nb;
    double phi = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
    double cm = 1.0, sm = 0.0, cp = 0.0, sp = 0.0;  // (x+iy)^m and (x+iy)^(m-1)
    double pmm = 1.0;
    for (int m = 0; m <= P; ++m) {
        if (m > 0) {
            cp = cm;
            sp = sm;
            double c2 = cm * x - sm * y;
            sm = sm * x + cm * y;
            cm = c2;
            pmm *= (2.0 * m - 1.0);
        }
        // Pi_{n-1}, Pi_{n-2} and their z / r2 derivatives
        double p1 = 0, p2 = 0, z1 = 0, z2 = 0, q1 = 0, q2 = 0;
        for (int n = m; n <= P; ++n) {
            double pn, dz, dq;
            if (n == m) {
                pn = pmm; dz = 0.0; dq = 0.0;
            } else if (n == m + 1) {
                pn = (2.0 * m + 1.0) * z * pmm;
                dz = (2.0 * m + 1.0) * pmm;
                dq = 0.0;
            } else {
                const double inv = 1.0 / (double)(n - m);
                pn = ((2.0 * n - 1.0) * z * p1 - (n + m - 1.0) * r2 * p2) * inv;
                dz = ((2.0 * n - 1.0) * (p1 + z * z1) - (n + m - 1.0) * r2 * z2) * inv;
                dq = ((2.0 * n - 1.0) * z * q1 - (n + m - 1.0) * (p2 + r2 * q2)) * inv;
            }
            p2 = p1; p1 = pn;
            z2 = z1; z1 = dz;
            q2 = q1; q1 = dq;
            // radial part gradient: dPi/dz e_z + 2 dPi/dr2 (x, y, z)
            const double rx = 2.0 * dq * x, ry = 2.0 * dq * y, rz = dz + 2.0 * dq * z;
            const int kc = n * n + n + m;
            const double ac = a[kc] * norm[kc];
            phi += ac * pn * cm;
            gx += ac * (pn * m * cp + cm * rx);
            gy += ac * (-pn * m * sp + cm * ry);
            gz += ac * (cm * rz);
            if (m > 0) {
                const int ks = n * n + n - m;
                const double as = a[ks] * norm[ks];
                phi += as * pn * sm;
                gx += as * (pn * m * sp + sm * rx);
                gy += as * (pn * m * cp + sm * ry);
                gz += as * (sm * rz);
            }
        }
    }
    const long long o = sd.part_off + i;
    phi_out[o] = phi;
    // gradient w.r.t. the scaled coordinates -> physical: times 1/Rs; E = -grad
    e_out[3 * o] = -gx * inv_rs;
    e_out[3 * o + 1] = -gy * inv_rs;
    e_out[3 * o + 2] = -gz * inv_rs;
}

}  // namespace

// FP32 form of series_field_kernel for the reduced precisions: the fully
// normalised recurrence (the coefficients of basis_df_tables, high words;
// every intermediate stays of order (r/Rs)^n, so no order leaves the FP32
// range) and its derivatives in z and r2,
//   d/dz  Pbar_n = a (Pbar_{n-1} + z d/dz Pbar_{n-1}) - b r2 d/dz Pbar_{n-2},
//   d/dr2 Pbar_n = a z d/dr2 Pbar_{n-1} - b (Pbar_{n-2} + r2 d/dr2 Pbar_{n-2}),
// in FP32 (positions from the split words, coefficients staged in shared
// memory), the sums over n folded into double-float accumulators after every
// m.  FP64 issue is slow on this part; this evaluates the fitted series at
// O(N N_b) FP32 cost.
__global__ void series_field_fp32_kernel(const __grid_constant__ BasisDfTables tabs, const SysDesc *sys, int nsys,
                                         int P, double inv_rs, const double *A, const float4 *src_hi,
                                         const float4 *src_lo, double *phi_out, double *e_out)
{
    extern __shared__ float ssm[];  // [Nb] coefficients A_k, a[m][n], b[m][n] ((P+1)^2 each), D, E
    const int s = blockIdx.y;
    const SysDesc sd = sys[s];
    const int W = P + 1, Nb = W * W;
    float *an = ssm, *ta = ssm + Nb, *tb = ta + W * W, *td = tb + W * W, *te = td + W;
    const double *a = A + (long long)s * Nb;
    for (int k = threadIdx.x; k < Nb; k += blockDim.x) {
        an[k] = (float)a[k];
        ta[k] = tabs.a[k / W][k % W].x;
        tb[k] = tabs.b[k / W][k % W].x;
    }
    for (int k = threadIdx.x; k <= P; k += blockDim.x) {
        td[k] = tabs.d[k].x;
        te[k] = tabs.e[k].x;
    }
    __syncthreads();
    const long long i = sd.sp_lo + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= sd.sp_lo + sd.sp_n) return;
    const float4 h = src_hi[sd.src_off + i], l = src_lo[sd.src_off + i];
    const float ir = (float)inv_rs;
    const float x = (h.x + l.x) * ir, y = (h.y + l.y) * ir, z = (h.z + l.z) * ir;
    const float r2 = fmaf(x, x, fmaf(y, y, z * z));
    float2 phi = make_float2(0.f, 0.f), gx = phi, gy = phi, gz = phi;
    float cm = 1.f, sm = 0.f, cp = 0.f, sp = 0.f;  // (x+iy)^m and (x+iy)^(m-1)
    for (int m = 0; m <= P; ++m) {
        if (m > 0) {
            cp = cm;
            sp = sm;
            const float c2 = cm * x - sm * y;
            sm = sm * x + cm * y;
            cm = c2;
        }
        const float fm = (float)m;
        float p1 = 0.f, p2 = 0.f, z1 = 0.f, z2 = 0.f, q1 = 0.f, q2 = 0.f;
        float fp = 0.f, fx = 0.f, fy = 0.f, fz = 0.f;
        const float *am = ta + m * W, *bm = tb + m * W;
        for (int n = m; n <= P; ++n) {
            float pn, dz, dq;
            if (n == m) {
                pn = td[m];
                dz = 0.f;
                dq = 0.f;
            } else if (n == m + 1) {
                pn = te[m] * z;
                dz = te[m];
                dq = 0.f;
            } else {
                const float ca = am[n], cb = bm[n];
                pn = ca * z * p1 - cb * r2 * p2;
                dz = ca * (p1 + z * z1) - cb * r2 * z2;
                dq = ca * z * q1 - cb * (p2 + r2 * q2);
            }
            p2 = p1; p1 = pn;
            z2 = z1; z1 = dz;
            q2 = q1; q1 = dq;
            const float rx = 2.f * dq * x, ry = 2.f * dq * y, rz = dz + 2.f * dq * z;
            const float ac = an[n * n + n + m];
            fp += ac * pn * cm;
            fx += ac * (pn * fm * cp + cm * rx);
            fy += ac * (-pn * fm * sp + cm * ry);
            fz += ac * (cm * rz);
            if (m > 0) {
                const float as = an[n * n + n - m];
                fp += as * pn * sm;
                fx += as * (pn * fm * sp + sm * rx);
                fy += as * (pn * fm * cp + sm * ry);
                fz += as * (sm * rz);
            }
        }
        phi = df_add(phi, fp);
        gx = df_add(gx, fx);
        gy = df_add(gy, fy);
        gz = df_add(gz, fz);
    }
    const long long o = sd.part_off + i;
    phi_out[o] = (double)phi.x + (double)phi.y;
    e_out[3 * o] = -((double)gx.x + (double)gx.y) * inv_rs;
    e_out[3 * o + 1] = -((double)gy.x + (double)gy.y) * inv_rs;
    e_out[3 * o + 2] = -((double)gz.x + (double)gz.y) * inv_rs;
}

int launch_series_field(const SysDesc *sys, int nsys, long long max_n, int P, double Rs, const double *norm,
                        const double *A, const float4 *src_hi, const float4 *src_lo, const double4_32a *src64,
                        double *phi_out, double *e_out, cudaStream_t st)
{
    dim3 grid((unsigned)((max_n + 127) / 128), nsys);
    if (!src64 && src_hi && P <= kBasisTableMaxP) {
        const size_t smem = sizeof(float) * (3 * (size_t)(P + 1) * (P + 1) + 2 * (size_t)(P + 1));
        series_field_fp32_kernel<<<grid, 128, smem, st>>>(basis_df_tables(), sys, nsys, P, 1.0 / Rs, A, src_hi, src_lo,
                                                          phi_out, e_out);
    } else {
        series_field_kernel<<<grid, 128, 0, st>>>(sys, nsys, P, 1.0 / Rs, norm, A, src_hi, src_lo, src64, phi_out,
                                                  e_out);
    }
    HSMA_LAUNCHED();
    HSMA_CUDA_TRY(cudaGetLastError());
    return HSMA_OK;
}

}  // namespace hsma
