// sc_reduce.cu -- cross-split reduction and FP64 epilogue of the FP32 path.
//
// The field kernels leave, per node table, split and (point, omega), the
// compensated float-float partials of the 12 sums of Sec. II Eq. 11's
// summand (E: U q + V z, B: Wv z) and a rim slot with the E sums of the
// boundary nodes.  reduce_lanes(n_splits) neighbouring threads share one
// (point, omega): each adds its run of splits as float-float pairs (TwoSum: an
// error of about 2^-47 of the largest partial, far below the FP32 result's
// last place), a shuffle tree adds the threads' sums the same way, and they
// share the components of the FP64 epilogue, which multiplies the rim sum by
// i/k_n (the factor of the line integral) and each node table's sum by its
// amplitude a_n w_p(omega_n):
//     E = sum_p amp_p (S_p + (i/k) rim_p),   B = sum_p amp_p S_p^B.
// The order depends on the request's split count alone, so results are
// deterministic and the same alone or in a batch.
//
// What bounds it: FP64 runs at 2 operations a cycle and SM here, and adding the
// splits in FP64 took four of them (two conversions, two additions) per value
// and split, one thread per (point, omega) in blocks of 256; now they are paid
// once per value and table.  Under ncu, cold caches: 1024 points x 1 omega x 64
// splits 230 -> 13 us (was 4 blocks, serial over the splits: latency), 3001 x 11
// x 48 splits 177 -> 48 us.  One lane per four splits: with one per sixteen the
// first took twice as long.
#include <cuda_runtime.h>

#include "sc_internal.h"

namespace sc {

namespace {

// Threads per (point, omega): 1, 2, 4 or 8, up to four splits each where that
// is possible.  They also share the six complex components of the epilogue.
__host__ __device__ inline int reduce_lanes(int n_splits)
{
    return n_splits <= 4 ? 1 : (n_splits <= 8 ? 2 : (n_splits <= 16 ? 4 : 8));
}

// threads of one request, whole warps
__host__ __device__ inline long long reduce_threads(int n_pts, int n_omega, int n_splits)
{
    return ((long long)n_pts * n_omega * reduce_lanes(n_splits) + 31) / 32 * 32;
}

// (h, l) += (a, b)
__device__ __forceinline__ void add_pair(float& h, float& l, float a, float b)
{
    const float t = h + a, v = t - h;
    l += ((h - (t - v)) + (a - v)) + b;
    h = t;
}

// Thread t of one request's reduction (whole warps reach this together).
template <int lanes>
__device__ __forceinline__ void reduce_lane(const ReduceLaunch& r, long long t)
{
    const long long idx = t / lanes;
    const int sub = (int)(t % lanes);
    const bool live = idx < (long long)r.n_pts * r.n_omega;
    const int pt = live ? (int)(idx / r.n_omega) : 0, n = live ? (int)(idx % r.n_omega) : 0;
    const size_t stride = (size_t)r.n_pts * r.n_omega * kAcc;
    const size_t at = ((size_t)pt * r.n_omega + n) * kAcc;
    // this thread's splits
    const int per = (r.n_splits + lanes - 1) / lanes;
    const int s0 = min(sub * per, r.n_splits), s1 = live ? min(s0 + per, r.n_splits) : s0;
    // each thread finishes the components c = sub, sub + lanes, ... of E_x .. B_z
    double re[6], im[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) re[j] = im[j] = 0.0;
    const double ik = 1.0 / r.kval[n];
    for (int p = 0; p < r.n_parts; ++p) {
        const float2* base = r.ws + (size_t)p * (r.n_splits + 1) * stride + at;
        float h[kAcc], l[kAcc];
#pragma unroll
        for (int c = 0; c < kAcc; ++c) h[c] = l[c] = 0.f;
#pragma unroll 4
        for (int sp = s0; sp < s1; ++sp) {
            const float4* v = reinterpret_cast<const float4*>(base + sp * stride);
#pragma unroll
            for (int c = 0; c < kAcc / 2; ++c) {
                const float4 q = __ldg(v + c);
                add_pair(h[2 * c], l[2 * c], q.x, q.y);
                add_pair(h[2 * c + 1], l[2 * c + 1], q.z, q.w);
            }
        }
#pragma unroll
        for (int o = 1; o < lanes; o *= 2)
#pragma unroll
            for (int c = 0; c < kAcc; ++c) {
                const float a = __shfl_xor_sync(0xffffffffu, h[c], o), b = __shfl_xor_sync(0xffffffffu, l[c], o);
                add_pair(h[c], l[c], a, b);
            }
        const float4* rim = reinterpret_cast<const float4*>(base + (size_t)r.n_splits * stride);
        const double ar = r.amp[p * r.amp_stride + 2 * n], ai = r.amp[p * r.amp_stride + 2 * n + 1];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const int c = sub + j * lanes;
            if (j * lanes >= 6) continue;
            // the sums of component c (selected: registers have no index)
            float sh = h[0], sl = l[0], th = h[1], tl = l[1];
#pragma unroll
            for (int i = 1; i < 6; ++i)
                if (c == i) sh = h[2 * i], sl = l[2 * i], th = h[2 * i + 1], tl = l[2 * i + 1];
            double tr = (double)sh + (isfinite(sh) ? (double)sl : 0.0);
            double ti = (double)th + (isfinite(th) ? (double)tl : 0.0);
            if (c < 3) {
                // T = S + (i/k) rim: the rim slot's E sum carries the factor i/k of
                // the line integral
                const float4 q = __ldg(rim + c);
                tr -= ik * ((double)q.z + (double)q.w);
                ti += ik * ((double)q.x + (double)q.y);
            }
            re[j] += ar * tr - ai * ti;  // the part adds amp_p T
            im[j] += ar * ti + ai * tr;
        }
    }
    if (!live) return;
    const size_t out = (size_t)n * r.out_pt_stride_omega + (size_t)pt * 3;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const int c = sub + j * lanes;
        const float2 v = make_float2((float)re[j], (float)im[j]);
        if (c < 3) r.E[out + c] = v;
        else if (c < 6 && r.B) r.B[out + c - 3] = v;
    }
}

__device__ __forceinline__ void reduce_one(const ReduceLaunch& r, long long t)
{
    switch (reduce_lanes(r.n_splits)) {
    case 1: return reduce_lane<1>(r, t);
    case 2: return reduce_lane<2>(r, t);
    case 4: return reduce_lane<4>(r, t);
    default: return reduce_lane<8>(r, t);
    }
}

// Small blocks, so that a reduction of a few thousand threads still reaches
// most SMs.
constexpr int kReduceBlock = 64;

__global__ void __launch_bounds__(kReduceBlock) reduce_kernel(ReduceLaunch r)
{
    reduce_one(r, (long long)blockIdx.x * kReduceBlock + threadIdx.x);
}

__global__ void __launch_bounds__(kReduceBlock) reduce_batch_kernel(const ReduceLaunch* reqs, int n_req,
                                                                    long long total)
{
    const long long t = (long long)blockIdx.x * kReduceBlock + threadIdx.x;
    if (t >= total) return;  // total counts whole warps
    int lo = 0, hi = n_req - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (reqs[mid].off <= t) lo = mid; else hi = mid - 1;
    }
    const ReduceLaunch& r = reqs[lo];
    reduce_one(r, t - r.off);
}

}  // namespace

long long reduce_size(const ReduceLaunch& r) { return reduce_threads(r.n_pts, r.n_omega, r.n_splits); }

int launch_reduce_f32(const ReduceLaunch& r, cudaStream_t s)
{
    const long long total = reduce_size(r);
    reduce_kernel<<<(unsigned)((total + kReduceBlock - 1) / kReduceBlock), kReduceBlock, 0, s>>>(r);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? 1 : -(int)e;
}

int launch_reduce_batch(const ReduceLaunch* reqs, int n_req, long long total, cudaStream_t s)
{
    if (total <= 0) return 0;
    reduce_batch_kernel<<<(unsigned)((total + kReduceBlock - 1) / kReduceBlock), kReduceBlock, 0, s>>>(reqs, n_req,
                                                                                                       total);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? 1 : -(int)e;
}

}  // namespace sc
