// sc_f64_idft.cu -- the plain FP64 field sum and the inverse transform of small
// sizes (sc_idft.cu has the tensor-core kernel of the others).
//
// field_f64_kernel: the same quadrature of Sec. II Eq. 11 as the FP32 kernel,
// in FP64 throughout, with the phase R - (z + 2f) + W formed by a direct
// difference.  It is both a second parity check and the FP64 GPU
// baseline.  An incident with several node tables runs once per table, the
// later ones adding to E and B.
//
// What bounds it: FP64 instructions, 2 a cycle and SM.  A term needs 21 of them
// (a phase factor's two forms and 18 sums); one thread per (point, omega) paid
// some 90 more for the pair's geometry (a square root, a division) and a sincos.
// Now gp threads of NB omegas share a point: each computes the pair of one node
// of every gp, and the first phase factor of every thread for it, into shared
// memory; all of them read it and go on from their first two factors by the
// three-term recurrence (on grids uniform to rounding; others take a sincos per
// omega).  Sine and cosine come from a table and short polynomials (16
// instructions).  512 points x 128^2 nodes x 64 omegas: 103.6 ms with a thread per
// (point, omega), 37.1 with shared pairs, a sincos per thread and rotations, now
// 30.2.  Where points and omegas are too few for the chip the nodes are split
// over the grid and the splits' sums added by a second kernel: 1024 points x
// 64^2 nodes x 1 omega, 8 blocks at first: 13.65 ms, 0.85 with splits, now 0.77.
//
// idft: Sec. III.B Eq. 13 for a real field sampled at positive k_n,
// F(t_m) = 2 dk Re sum_n F_n e^{-i k_n t_m}, as a phasor table
// M[n][m] = e^{-i k_n t_m} (built in FP64, stored as float2) contracted with
// the spectra by a shared-memory tiled FP32 kernel.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "sc_internal.h"

namespace sc {

namespace {

constexpr int kF64Threads = 128;
constexpr int kF64Row = 13;  // doubles per shared pair row: ir, phi, U, V, Wv, rotation e^{i dk Phi}
                             // (and then the threads' first phase factors)

// sin and cos by table lookup (P. T. P. Tang, "Table-lookup algorithms for
// elementary functions and their error analysis", 1991): x = j 2 pi / N + r with
// |r| <= pi / N, the N pairs (cos, sin)(2 pi j / N) from memory and Taylor
// polynomials of sin r and cos r - 1 (the first terms left out are below 2^-59 for
// N = 1024).  16 FP64 instructions; sincos() takes about 37.  Arguments from 2^30
// on, infinities and NaN go to sincos().
constexpr int kTrigN = kTrigEntries;
constexpr double kTrigStepLo = 2.391888279584674e-19;  // 2 pi / N beyond its double

__device__ __forceinline__ void sincos_tab(const double2* tab, double x, double* sn, double* cs)
{
    if ((__double2hiint(x) & 0x7fffffff) >= 0x41d00000) {
        sincos(x, sn, cs);
        return;
    }
    constexpr double kMagic = 6755399441055744.0;  // 1.5 2^52: the sum's low bits are the nearest integer
    const double t = fma(x, 162.97466172610083, kMagic);  // N / (2 pi)
    const double j = t - kMagic;
    double r = fma(j, -0.006135923151542565, x);           // 2 pi / N, and what the double leaves of it
    r = fma(j, -kTrigStepLo, r);
    const double2 cS = __ldg(tab + (__double2loint(t) & (kTrigN - 1)));
    const double r2 = r * r;
    const double sr = fma(r * r2, fma(r2, 1.0 / 120.0, -1.0 / 6.0), r);
    const double cm = r2 * fma(r2, 1.0 / 24.0, -0.5);
    *sn = cS.y + fma(cS.y, cm, cS.x * sr);
    *cs = cS.x + fma(cS.x, cm, -cS.y * sr);
}

__global__ void trig_table_kernel(double2* tab)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= kTrigN) return;
    double s, c;
    sincospi(2.0 * j / kTrigN, &s, &c);
    tab[j] = make_double2(c, s);
}

// One pair's geometry: row = {1/R, Phi, U[3], V[3], Wv[3]}.
__device__ __forceinline__ void pair64(const Node64& nd, double x, double y, double z, double row[11])
{
    const double dx = nd.px - x, dy = nd.py - y, dz = nd.pz - z;
    const double R = sqrt(dx * dx + dy * dy + dz * dz);
    const double ir = 1.0 / R;
    const double rx = dx * ir, ry = dy * ir, rz = dz * ir;
    const double ux = nd.jx * ir, uy = nd.jy * ir, uz = nd.jz * ir;
    const double av = nd.rho * ir;
    row[0] = ir;
    row[1] = (R - nd.pn) + nd.w;
    row[2] = ux; row[3] = uy; row[4] = uz;
    row[5] = av * rx; row[6] = av * ry; row[7] = av * rz;
    row[8] = uy * rz - uz * ry;
    row[9] = uz * rx - ux * rz;
    row[10] = ux * ry - uy * rx;
}

// Without the common factor ik: E' += U ph + V y, B' += Wv y with ph = (c, s) and
// y = (1 + i / (kR)) ph; w = 1 / (kR).
__device__ __forceinline__ void eval64(double sE[6], double sB[6], const double* row, double ik, double c, double s)
{
    const double w = row[0] * ik;
    const double yr = c - w * s, yi = s + w * c;
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) {
        sE[2 * cc] += row[2 + cc] * c + row[5 + cc] * yr;
        sE[2 * cc + 1] += row[2 + cc] * s + row[5 + cc] * yi;
        sB[2 * cc] += row[8 + cc] * yr;
        sB[2 * cc + 1] += row[8 + cc] * yi;
    }
}

// ik times a node range's sums
__device__ __forceinline__ void times_ik(double s[6], double k)
{
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) {
        // (rounded: a sum of several node ranges must not contract the product into its addition)
        const double re = s[2 * cc];
        s[2 * cc] = __dmul_rn(-k, s[2 * cc + 1]);
        s[2 * cc + 1] = __dmul_rn(k, re);
    }
}

// The outputs of one (point, omega) from its surface sums and rim E sums:
// amp (S + (i/k) rim); later table parts add to the earlier ones.
__device__ __forceinline__ void finish64(const Field64Launch& a, int n, int pt, const double sE[6],
                                         const double sB[6], const double sR[6], int accumulate)
{
    const double ar = a.amp[2 * n], ai = a.amp[2 * n + 1], ik = 1.0 / a.kval[n];
    double2* E = a.E + ((size_t)n * a.n_pts + pt) * 3;
    for (int cc = 0; cc < 3; ++cc) {
        const double er = sE[2 * cc] - ik * sR[2 * cc + 1];
        const double ei = sE[2 * cc + 1] + ik * sR[2 * cc];
        double2 v = make_double2(ar * er - ai * ei, ar * ei + ai * er);
        if (accumulate) v = make_double2(v.x + E[cc].x, v.y + E[cc].y);
        E[cc] = v;
    }
    if (a.B) {
        double2* B = a.B + ((size_t)n * a.n_pts + pt) * 3;
        for (int cc = 0; cc < 3; ++cc) {
            const double br = sB[2 * cc], bi = sB[2 * cc + 1];
            double2 v = make_double2(ar * br - ai * bi, ar * bi + ai * br);
            if (accumulate) v = make_double2(v.x + B[cc].x, v.y + B[cc].y);
            B[cc] = v;
        }
    }
}

// Sum the nodes [j0, j1) into NB omegas' E and B.  gp threads (neighbouring
// lanes, a power of two) of a point share its pairs through rows, `stride` doubles
// each: kF64Row of the pair and, with UNI, 2 gp of the threads' first phase factors.
template <int NB, bool UNI>
__device__ __forceinline__ void sum64(const Field64Launch& a, const Node64* nodes, int j0, int j1, double x, double y,
                                      double z, int g, double k0, const double kv[NB], const double ikv[NB],
                                      double* rows, int stride, double (*sE)[6], double (*sB)[6])
{
#pragma unroll
    for (int i = 0; i < NB; ++i)
#pragma unroll
        for (int c = 0; c < 6; ++c) sE[i][c] = sB[i][c] = 0.0;
    double* mine = rows + threadIdx.x * stride;
    const double* base = rows + (threadIdx.x - g) * stride;  // the point's first row
    for (int j = j0; j < j1; j += a.gp) {
        double own[kF64Row];
        double fs = 0.0, fc = 1.0;  // own first phase factor (gp = 1)
        if (a.gp > 1) __syncwarp();  // the last round's rows are read
        if (j + g < j1) {
            pair64(nodes[j + g], x, y, z, own);
            if (NB > 1 && UNI) sincos_tab(a.trig, a.dk * own[1], &own[12], &own[11]);
            if (a.gp > 1) {
#pragma unroll
                for (int i = 0; i < kF64Row; ++i)
                    if (i < 11 || (NB > 1 && UNI)) mine[i] = own[i];
                if (UNI) {
                    // e^{i (k0 + h NB dk) Phi} for every thread h of the point, by rotation
                    // (k0: the first omega of the point's first thread)
                    double rs, rc;
                    sincos_tab(a.trig, k0 * own[1], &fs, &fc);
                    sincos_tab(a.trig, NB * a.dk * own[1], &rs, &rc);
                    for (int h = 0; h < a.gp; ++h) {
                        reinterpret_cast<double2*>(mine + kF64Row + 1)[h] = make_double2(fc, fs);
                        const double t = fc * rc - fs * rs;
                        fs = fc * rs + fs * rc;
                        fc = t;
                    }
                }
            } else {
                sincos_tab(a.trig, kv[0] * own[1], &fs, &fc);
            }
        }
        const int m = min(a.gp, j1 - j);
        if (a.gp > 1) __syncwarp();
        for (int q = 0; q < m; ++q) {
            double row[kF64Row];
            if (a.gp > 1) {
                const double* r = base + q * stride;
#pragma unroll
                for (int i = 0; i < kF64Row; ++i)
                    if (i < 11 || (NB > 1 && UNI)) row[i] = r[i];
                if (UNI) {
                    const double2 f = reinterpret_cast<const double2*>(r + kF64Row + 1)[g];
                    fc = f.x;
                    fs = f.y;
                } else {
                    sincos_tab(a.trig, kv[0] * row[1], &fs, &fc);
                }
            } else {
#pragma unroll
                for (int i = 0; i < kF64Row; ++i) row[i] = own[i];
            }
            eval64(sE[0], sB[0], row, ikv[0], fc, fs);
            if (UNI && NB > 1) {
                double c0 = fc, s0 = fs;
                double c1 = fc * row[11] - fs * row[12], s1 = fc * row[12] + fs * row[11];
                const double two = 2.0 * row[11];
#pragma unroll
                for (int i = 1; i < NB; ++i) {
                    eval64(sE[i], sB[i], row, ikv[i], c1, s1);
                    if (i + 1 < NB) {
                        const double c2 = fma(two, c1, -c0), s2 = fma(two, s1, -s0);
                        c0 = c1;
                        s0 = s1;
                        c1 = c2;
                        s1 = s2;
                    }
                }
            } else {
#pragma unroll
                for (int i = 1; i < NB; ++i) {
                    double s, c;
                    sincos_tab(a.trig, kv[i] * row[1], &s, &c);
                    eval64(sE[i], sB[i], row, ikv[i], c, s);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        times_ik(sE[i], kv[i]);
        times_ik(sB[i], kv[i]);
    }
}

// doubles of a shared row; a row's phase factors start on 16 bytes
__host__ __device__ inline int f64_stride(int gp) { return gp > 1 ? kF64Row + 1 + 2 * gp : 0; }

// blockIdx.x: points (128 / gp of them), y: omegas (gp NB of them), z: node
// split.  One split sums surface and rim and writes the outputs; with several,
// split z < n_splits writes its share's 12 sums to ws and z = n_splits the
// rim's.  SERIAL: the several splits of a call that has no room for ws, one after
// another, added and finished in the order of reduce_f64_kernel, so that a result's
// bits do not depend on the room there was.
template <int NB, bool UNI, bool SERIAL>
__global__ void __launch_bounds__(kF64Threads) field_f64_kernel(Field64Launch a)
{
    extern __shared__ __align__(16) double rows[];
    const int stride = f64_stride(a.gp);
    const int g = threadIdx.x % a.gp;
    const int pt = blockIdx.x * (kF64Threads / a.gp) + threadIdx.x / a.gp;
    const int n0 = (blockIdx.y * a.gp + g) * NB;
    const bool live = pt < a.n_pts;  // (idle lanes follow: their warp shares rows)
    const int p = live ? pt : a.n_pts - 1;
    const double x = a.pts[3 * p], y = a.pts[3 * p + 1], z = a.pts[3 * p + 2];
    const double k0 = a.kval[min((int)blockIdx.y * a.gp * NB, a.n_omega - 1)];
    double kv[NB], ikv[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        kv[i] = a.kval[min(n0 + i, a.n_omega - 1)];
        ikv[i] = 1.0 / kv[i];
    }
    double sE[NB][6], sB[NB][6];
    if constexpr (SERIAL) {
        double tE[NB][6] = {}, tB[NB][6] = {};
        const int per = (a.n_surf + a.n_splits - 1) / a.n_splits;
        for (int sp = 0; sp < a.n_splits; ++sp) {
            const int j0 = min(sp * per, a.n_surf);
            sum64<NB, UNI>(a, a.surf, j0, min(j0 + per, a.n_surf), x, y, z, g, k0, kv, ikv, rows, stride, sE, sB);
#pragma unroll
            for (int i = 0; i < NB; ++i)
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    tE[i][c] += sE[i][c];
                    tB[i][c] += sB[i][c];
                }
        }
        sum64<NB, UNI>(a, a.rim, 0, a.n_rim, x, y, z, g, k0, kv, ikv, rows, stride, sE, sB);
        if (live)
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (n0 + i < a.n_omega) finish64(a, n0 + i, pt, tE[i], tB[i], sE[i], a.accumulate);
        return;
    }
    if (a.n_splits > 1) {
        const bool rim = (int)blockIdx.z == a.n_splits;
        const int per = (a.n_surf + a.n_splits - 1) / a.n_splits;
        const int j0 = rim ? 0 : min((int)blockIdx.z * per, a.n_surf);
        sum64<NB, UNI>(a, rim ? a.rim : a.surf, j0, rim ? a.n_rim : min(j0 + per, a.n_surf), x, y, z, g, k0, kv, ikv,
                       rows, stride, sE, sB);
        if (!live) return;
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (n0 + i < a.n_omega) {
                double* w = a.ws + (((size_t)blockIdx.z * a.n_omega + n0 + i) * a.n_pts + pt) * kAcc;
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    w[c] = sE[i][c];
                    w[6 + c] = sB[i][c];
                }
            }
        return;
    }
    // one split: the rim's part of the outputs, then the surface's added to it
    const double zero[6] = {0, 0, 0, 0, 0, 0};
    sum64<NB, UNI>(a, a.rim, 0, a.n_rim, x, y, z, g, k0, kv, ikv, rows, stride, sE, sB);
    if (live)
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (n0 + i < a.n_omega) finish64(a, n0 + i, pt, zero, zero, sE[i], a.accumulate);
    sum64<NB, UNI>(a, a.surf, 0, a.n_surf, x, y, z, g, k0, kv, ikv, rows, stride, sE, sB);
    if (live)
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (n0 + i < a.n_omega) finish64(a, n0 + i, pt, sE[i], sB[i], zero, 1);
}

// The splits' sums in split order, and the outputs: 12 threads per (point,
// omega), one sum each, then one of them finishes.
constexpr int kF64Red = 16;  // (point, omega) entries per block

__global__ void __launch_bounds__(12 * kF64Red) reduce_f64_kernel(Field64Launch a)
{
    __shared__ double sums[kF64Red][18];
    const int e = threadIdx.x / 12, c = threadIdx.x % 12;
    const long long idx = (long long)blockIdx.x * kF64Red + e;
    const bool live = idx < (long long)a.n_pts * a.n_omega;
    if (live) {
        const size_t stride = (size_t)a.n_pts * a.n_omega * kAcc;
        const double* w = a.ws + (size_t)idx * kAcc + c;
        double s = 0.0;
#pragma unroll 8
        for (int sp = 0; sp < a.n_splits; ++sp) s += w[sp * stride];
        sums[e][c] = s;
        if (c < 6) sums[e][12 + c] = w[a.n_splits * stride];
    }
    __syncthreads();
    if (live && c == 0)
        finish64(a, (int)(idx / a.n_pts), (int)(idx % a.n_pts), sums[e], sums[e] + 6, sums[e] + 12,
                 a.accumulate);
}

__global__ void phasor_kernel(const double* kval, int n_omega, const double* t, int n_t,
                              float2* M)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)n_omega * n_t) return;
    const int n = (int)(idx / n_t), m = (int)(idx % n_t);
    double s, c;
    sincos(kval[n] * t[m], &s, &c);
    M[idx] = make_float2((float)c, (float)-s);
}

__device__ __forceinline__ float2 load_c(const float2* F, size_t i) { return F[i]; }
__device__ __forceinline__ float2 load_c(const double2* F, size_t i)
{
    const double2 v = F[i];
    return make_float2((float)v.x, (float)v.y);
}

// out[m][v] = scale * sum_n Re(F[n][v] M[n][m]); 64 x 64 output tile per
// CTA (16 x 16 threads, 4 x 4 outputs each), 8 frequencies per smem stage.
template <typename T>
__global__ void __launch_bounds__(256) idft_kernel(const T* F, int n_omega, long long n_vals,
                                                   const float2* M, int n_t, float scale,
                                                   float* out, int accumulate)
{
    __shared__ float2 Ms[8][64];
    __shared__ float2 Fs[8][64];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int m0 = blockIdx.y * 64;
    const long long v0 = (long long)blockIdx.x * 64;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int n0 = 0; n0 < n_omega; n0 += 8) {
        for (int e = threadIdx.x; e < 8 * 64; e += 256) {
            const int nn = e / 64, c = e % 64;
            const int n = n0 + nn;
            const int m = m0 + c;
            const long long v = v0 + c;
            Ms[nn][c] = (n < n_omega && m < n_t) ? M[(size_t)n * n_t + m] : make_float2(0.f, 0.f);
            Fs[nn][c] = (n < n_omega && v < n_vals) ? load_c(F, (size_t)n * n_vals + v)
                                                    : make_float2(0.f, 0.f);
        }
        __syncthreads();
#pragma unroll
        for (int nn = 0; nn < 8; ++nn) {
            float2 mv[4], fv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) mv[i] = Ms[nn][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) fv[j] = Fs[nn][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc[i][j] = fmaf(fv[j].x, mv[i].x, fmaf(-fv[j].y, mv[i].y, acc[i][j]));
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty + 16 * i;
        if (m >= n_t) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long v = v0 + tx + 16 * j;
            if (v < n_vals) {
                float* o = out + (size_t)m * n_vals + v;
                *o = accumulate ? *o + scale * acc[i][j] : scale * acc[i][j];
            }
        }
    }
}

}  // namespace

namespace {

using F64Kernel = void (*)(Field64Launch);

template <bool SERIAL>
F64Kernel f64_kernel(int nb, bool uni)
{
    switch (nb) {
    case 1: return field_f64_kernel<1, false, SERIAL>;
    case 2: return uni ? field_f64_kernel<2, true, SERIAL> : field_f64_kernel<2, false, SERIAL>;
    case 3: return uni ? field_f64_kernel<3, true, SERIAL> : field_f64_kernel<3, false, SERIAL>;
    case 4: return uni ? field_f64_kernel<4, true, SERIAL> : field_f64_kernel<4, false, SERIAL>;
    case 5: return uni ? field_f64_kernel<5, true, SERIAL> : field_f64_kernel<5, false, SERIAL>;
    default: return uni ? field_f64_kernel<6, true, SERIAL> : field_f64_kernel<6, false, SERIAL>;
    }
}

}  // namespace

void plan_field_f64(Field64Launch& a, int device)
{
    // threads per point and omegas per thread: as few threads of up to six
    // omegas (twelve FP64 sums each: more spill) as cover the omegas, at most
    // 32, whose omegas then come out even
    a.gp = 1;
    while (a.gp < 32 && a.n_omega > 6 * a.gp) a.gp *= 2;
    a.nb = a.n_omega >= 6 * a.gp ? 6 : (a.n_omega + a.gp - 1) / a.gp;
    int per_sm = 1, sms = 1;
    const size_t smem = (size_t)kF64Threads * f64_stride(a.gp) * sizeof(double);
    const F64Kernel kern = f64_kernel<false>(a.nb, a.dk > 0.0);
    if (smem > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kF64Threads, smem) != cudaSuccess) per_sm = 1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) sms = 1;
    cudaGetLastError();
    const int slots = std::max(1, per_sm) * std::max(1, sms);
    const long long blocks = (long long)((a.n_pts + kF64Threads / a.gp - 1) / (kF64Threads / a.gp)) *
                             ((a.n_omega + a.gp * a.nb - 1) / (a.gp * a.nb));
    // node splits: none from four waves of blocks on; below that about four
    // waves, of at least 32 nodes and two rounds of gp
    long long s = blocks >= 4LL * slots ? 1 : (4LL * slots + blocks - 1) / blocks;
    s = std::min<long long>(s, std::max(1, a.n_surf / std::max(32, 2 * a.gp)));
    a.n_splits = (int)std::min<long long>(s, 1024);
}

int launch_trig_table(double2* tab, cudaStream_t s)
{
    trig_table_kernel<<<kTrigN / 128, 128, 0, s>>>(tab);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? 1 : -(int)e;
}

size_t field_f64_workspace(const Field64Launch& a)
{
    return a.n_splits > 1 ? (size_t)(a.n_splits + 1) * a.n_omega * a.n_pts * kAcc * sizeof(double) : 0;
}

int launch_field_f64(const Field64Launch& a, cudaStream_t s)
{
    const int ppb = kF64Threads / a.gp, opb = a.gp * a.nb;
    const dim3 grid((unsigned)((a.n_pts + ppb - 1) / ppb), (unsigned)((a.n_omega + opb - 1) / opb),
                    (unsigned)(a.ws ? a.n_splits + 1 : 1));
    const size_t smem = (size_t)kF64Threads * f64_stride(a.gp) * sizeof(double);
    const bool serial = a.n_splits > 1 && !a.ws;
    const F64Kernel kern = serial ? f64_kernel<true>(a.nb, a.dk > 0.0) : f64_kernel<false>(a.nb, a.dk > 0.0);
    cudaError_t e = cudaSuccess;
    if (serial && smem > 48 * 1024)  // (plan_field_f64 raised the other's limit)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return -(int)e;
    kern<<<grid, kF64Threads, smem, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return -(int)e;
    if (!a.ws) return 1;
    const long long total = (long long)a.n_pts * a.n_omega;
    reduce_f64_kernel<<<(unsigned)((total + kF64Red - 1) / kF64Red), 12 * kF64Red, 0, s>>>(a);
    e = cudaGetLastError();
    return e == cudaSuccess ? 2 : -(int)e;
}

int launch_idft(const IdftLaunch& p, cudaStream_t s)
{
    const long long nm = (long long)p.n_omega * p.n_t;
    phasor_kernel<<<(unsigned)((nm + 255) / 256), 256, 0, s>>>(p.kval, p.n_omega, p.t, p.n_t,
                                                               p.phasor);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return -(int)e;
    dim3 grid((unsigned)((p.n_vals + 63) / 64), (unsigned)((p.n_t + 63) / 64));
    const float scale = (float)(2.0 * p.dk);
    if (p.f64)
        idft_kernel<double2><<<grid, 256, 0, s>>>((const double2*)p.F, p.n_omega, p.n_vals,
                                                  p.phasor, p.n_t, scale, p.out, p.accumulate);
    else
        idft_kernel<float2><<<grid, 256, 0, s>>>((const float2*)p.F, p.n_omega, p.n_vals,
                                                 p.phasor, p.n_t, scale, p.out, p.accumulate);
    e = cudaGetLastError();
    return e == cudaSuccess ? 2 : -(int)e;
}

}  // namespace sc
