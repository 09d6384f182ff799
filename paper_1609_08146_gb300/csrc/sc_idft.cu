// sc_idft.cu -- the inverse transform of Sec. III.B, Eq. 13 on the tensor
// cores: for a real field sampled at positive k_n,
//     out[m][v] = 2 dk Re sum_n F[n][v] e^{-i k_n t_m}
//               = 2 dk sum_n (Re F[n][v] cos k_n t_m + Im F[n][v] sin k_n t_m),
// a product of the phase table [times][2 omegas] with the spectra [2 omegas]
// [values].  (sc_f64_idft.cu keeps the FP32 kernel for small transforms.)
//
// Precision.  As in sc_field_tensor.cu both operands are split into two fp16
// halves and three products are accumulated (hi hi apart from hi lo + lo hi) in
// runs of kRunStages stages of 16 omegas, which are read, given back the
// expected loss of the tensor cores' truncation and added in FP32 registers.  The
// spectra are scaled by a power of two per value (column), from its largest
// entry, so that a value's rounding is relative to its own size.  A value with an
// infinity or a NaN is left to a plain FP32 loop.  Phases are formed in FP64.
//
// What bounds it.  4160 points x 3 components x 256 omegas -> 512 times, E and B:
// 102 MB in and out (15 us at the copy rate), 13 GFLOP (times three products: 21
// us at the measured tensor rate).  The FP32 kernel took 2 x 208 us plus the
// table twice; this one about 78 us and 12 for the table and scales, 436 -> 96 us
// the call.  What is left is mostly L2: every CTA reads its 256 times of the phase
// table (32 KB a stage beside 16 KB of spectra, 392 x 16 stages: 308 MB in all at
// about 4 TB/s); then the stores and the waves' tail (392 CTAs on 152 SMs).
//
// Structure: a CTA makes 128 values x MT 128 times of one field (16 warps):
//   warps 0-7   MT sets of four read their 128 times' accumulator (TMEM, all 512
//               columns for MT = 2) after every run and keep the sums in
//               registers; at the end they scale, transpose through shared
//               memory and store;
//   warp 8      issues the MMAs; warp 9 copies the phase table's stages (bulk
//               copies, the table is built once per transform in stage layout);
//   warps 12-15 convert the spectra's stages.
// A first kernel makes the phase table and the values' scales.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "sc_field_common.cuh"
#include "sc_internal.h"
#include "sc_tensor.cuh"

namespace sc {

namespace {

constexpr int kIM = 128;                    // times per accumulator
constexpr int kIV = 128;                    // values per CTA
constexpr int kIOm = 16;                    // omegas per stage (K = 32: real and imaginary parts)
constexpr int kAHalf = kIM * 2 * kIOm * 2;  // one half of a stage of the phase table: 8 KB
constexpr int kBHalf = kIV * 2 * kIOm * 2;  // one half of a stage of the spectra: 8 KB
constexpr int kRunStages = 3;
constexpr int kRawBytes = 64 * 1024;        // spectra on their way: 4 stages of FP32, 2 of FP64
constexpr int kIThreads = 512;
constexpr int kIEpiRegs = 168, kIOtherRegs = 88;
static_assert(256 * kIEpiRegs + 256 * kIOtherRegs <= 65536, "register split");

template <int MT>
struct Idft {
    static constexpr int STAGE = MT * 2 * kAHalf + 2 * kBHalf;
    static constexpr int STAGES = 3;
    static constexpr int OFF_RAW = STAGES * STAGE;            // spectra as they are, kRawBytes
    static constexpr int OFF_SCALE = OFF_RAW + kRawBytes;          // float scale[kIV]
    static constexpr int OFF_BAR = OFF_SCALE + kIV * 4;
    static constexpr int SMEM = OFF_BAR + 256;
    static constexpr int ACC = 2 * kIV;                       // columns of one accumulator: hi hi, then the rest
    static constexpr int ALLOC = MT * ACC;
    static_assert(SMEM <= 227 * 1024, "shared memory");
    static_assert(MT * 4 * 32 * (kIV + 1) * 4 <= STAGES * STAGE + kRawBytes, "transpose");
};

// The phase table in stage layout: for every 128 times and 16 omegas the high
// halves, then the low halves, of [times][K], K = 2 n (cosine), 2 n + 1 (sine);
// K-major: 16 bytes hold four omegas of one time.  One thread per time and stage:
// a sincos in FP64 for its first omega and (where the grid is uniform to
// rounding) rotations for the others.
constexpr int kAKStep = kIM * 16;      // bytes between blocks of 8 K
constexpr int kBKStep = 2 * kIV * 16;  // the spectra's: 128 values' high halves, then the low ones

__device__ __forceinline__ void table_stage(const IdftLaunch& p, int mb, int stage, int n_stages)
{
    const int m = mb * kIM + threadIdx.x;
    unsigned char* out = p.table + ((size_t)mb * n_stages + stage) * 2 * kAHalf;
    const double tm = m < p.n_t ? p.t[m] : 0.0;
    const int n0 = stage * kIOm;
    double s = 0.0, c = 1.0, rs = 0.0, rc = 1.0;
    if (p.dk_rot > 0.0) sincos(p.dk_rot * tm, &rs, &rc);
#pragma unroll
    for (int b = 0; b < kIOm / 4; ++b) {
        float2 x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int n = n0 + b * 4 + i;
            if (n == n0 || !(p.dk_rot > 0.0)) {
                sincos(p.kval[min(n, p.n_omega - 1)] * tm, &s, &c);
            } else {
                const double u = c * rc - s * rs;
                s = c * rs + s * rc;
                c = u;
            }
            x[i] = n < p.n_omega && m < p.n_t ? make_float2((float)c, (float)s) : make_float2(0.f, 0.f);
        }
        unsigned char* q = out + b * kAKStep + threadIdx.x * 16;
        split_store8(q, q + kAHalf, x);
    }
}

__device__ __forceinline__ float2 load_f32(const float2* F, size_t i) { return F[i]; }
__device__ __forceinline__ float2 load_f32(const double2* F, size_t i)
{
    const double2 v = F[i];
    return make_float2((float)v.x, (float)v.y);
}

// Cosine and sine of k t for a product with an infinity: right in sign and where they
// are zero.  In FP32 after a reduction in FP64, except near a zero.
__device__ __forceinline__ float2 sign_phase(double k, double t)
{
    const double u = k * t, q = u * 0.15915494309189535;
    float s, c;
    sincospif((float)(2.0 * (q - rint(q))), &s, &c);
    if (!(fabs(u) < 1e8) || (t != 0.0 && fminf(fabsf(c), fabsf(s)) < 1e-5f)) {
        double sd, cd;
        sincos(u, &sd, &cd);
        return make_float2((float)cd, (float)sd);
    }
    return make_float2(c, s);
}

// Before the product: blocks below n_table make a stage of the phase table each
// (FP64 latency), the others scan 32 values (columns) for their largest entry
// (memory latency), a power of two of which scales them into [2^11, 2^12); 0 marks
// a value with an infinity or a NaN.  One launch, so that either hides the other.
// The exponent spans -116 (entries from 2^127) to 126, the largest whose inverse
// is normal: entries below 2^-115, subnormal ones among them, come out smaller than
// 2^11, but all their bits still fit the two halves, whose last place is 2^-24 at
// most (an entry of 2^-149 scales to 2^-23).
constexpr int kScanCols = 32;

template <typename T>
__global__ void __launch_bounds__(kIM) idft_prep_kernel(const __grid_constant__ IdftLaunch p, int n_stages, int n_table)
{
    if ((int)blockIdx.x < n_table) return table_stage(p, blockIdx.x / n_stages, blockIdx.x % n_stages, n_stages);
    __shared__ int part[kIM / kScanCols][kScanCols];
    const long long blocks = (p.n_vals + kScanCols - 1) / kScanCols;
    const long long blk = (long long)blockIdx.x - n_table;
    const int field = blk >= blocks;
    const T* F = reinterpret_cast<const T*>(field ? p.F2 : p.F);
    const int c = threadIdx.x % kScanCols, q = threadIdx.x / kScanCols;
    const long long v = (blk - field * blocks) * kScanCols + c;
    // as bits, which order like the non-negative floats, infinities and NaN above
    int mx = 0;
    if (v < p.n_vals)
#pragma unroll 16
        for (int n = q; n < p.n_omega; n += kIM / kScanCols) {
            const float2 f = load_f32(F, (size_t)n * p.n_vals + v);
            mx = max(mx, max(__float_as_int(fabsf(f.x)), __float_as_int(fabsf(f.y))));
        }
    part[q][c] = mx;
    __syncthreads();
    if (q > 0 || v >= p.n_vals) return;
#pragma unroll
    for (int i = 1; i < kIM / kScanCols; ++i) mx = max(mx, part[i][c]);
    const float f = __int_as_float(mx);
    const int e = f > 0.f && f < INFINITY ? min(11 - ilogbf(f), 126) : 0;
    p.col_scale[field * p.n_vals + v] = mx >= 0x7f800000 ? 0.f : ldexpf(1.f, e);
}

// A warp's 32 times of the values with an infinity or a NaN (plain: 128 bits), lane =
// time.  Finite entries do not change such a sum, so the warp looks for the others,
// lane = omega, and adds them until every time's sum is NaN, which nothing changes any
// more; where fewer times are left than entries, lanes change over.  256 omegas, 4160
// points, 512 times, E and B: no such value 0.10 ms, one entry in 2% of the values
// 0.16, one in each 1.3, E infinite and B NaN throughout 11 (a sincos for every entry
// and time: 6.5, 189 and 189 ms; the FP32 kernel: 0.45).  A function of its own:
// inlined, the transform without such values took 2% longer.
template <typename T>
__device__ __noinline__ void plain_values(const IdftLaunch& p, const T* F, float* out, long long v0, int nv, int mw,
                                          const unsigned* plain)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kGroups = 8;  // of 32 omegas, whose loads are in flight together
    const int lane = threadIdx.x & 31;
    const int rows = min(32, p.n_t - mw);
    if (rows <= 0) return;
    const double tm = lane < rows ? p.t[mw + lane] : 0.0;
    for (int c = 0; c < nv; ++c) {
        if ((c & 31) == 0 && plain[c >> 5] == 0) {
            c += 31;
            continue;
        }
        if (!(plain[c >> 5] >> (c & 31) & 1)) continue;
        float a = 0.f;
        unsigned open = kAll >> (32 - rows);  // times whose sum is not NaN yet
        for (int n0 = 0; n0 < p.n_omega && open; n0 += 32 * kGroups) {
            float2 f[kGroups];
#pragma unroll
            for (int i = 0; i < kGroups; ++i) {
                const int n = n0 + 32 * i + lane;
                f[i] = n < p.n_omega ? load_f32(F + v0 + c, (size_t)n * p.n_vals) : make_float2(0.f, 0.f);
            }
#pragma unroll 1
            for (int i = 0; i < kGroups; ++i) {
                const float2 v = f[0];
#pragma unroll
                for (int j = 0; j + 1 < kGroups; ++j) f[j] = f[j + 1];
                const bool bad = !(isfinite(v.x) && isfinite(v.y));
                unsigned found = __ballot_sync(kAll, bad);
                while (found && open) {
                    if (__popc(found) <= __popc(open)) {  // one entry, lane = time
                        const int at = __ffs(found) - 1;
                        found &= found - 1;
                        const float2 ph = sign_phase(p.kval[n0 + 32 * i + at], tm);
                        a = fmaf(__shfl_sync(kAll, v.x, at), ph.x, fmaf(__shfl_sync(kAll, v.y, at), ph.y, a));
                    } else {  // every entry for each time that is left, lane = omega
                        for (unsigned left = open; left; left &= left - 1) {
                            const int at = __ffs(left) - 1;
                            const float2 ph = sign_phase(p.kval[min(n0 + 32 * i + lane, p.n_omega - 1)],
                                                         __shfl_sync(kAll, tm, at));
                            float u = bad ? fmaf(v.x, ph.x, v.y * ph.y) : 0.f;
                            for (int o = 16; o; o >>= 1) u += __shfl_xor_sync(kAll, u, o);
                            if (lane == at) a += u;
                        }
                        found = 0;
                    }
                    open &= __ballot_sync(kAll, !isnan(a));
                }
            }
        }
        if (lane >= rows) continue;
        float* o = out + (size_t)(mw + lane) * p.n_vals + v0 + c;
        *o = p.accumulate ? *o + p.scale * a : p.scale * a;
    }
}

template <typename T, int MT>
__global__ void __launch_bounds__(kIThreads, 1) idft_tensor_kernel(const __grid_constant__ IdftLaunch p, int n_stages)
{
    using L = Idft<MT>;
    extern __shared__ __align__(1024) unsigned char smem[];
    float* scale = reinterpret_cast<float*>(smem + L::OFF_SCALE);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR);  // [STAGES]
    uint64_t* tfull = full + L::STAGES;                               // [STAGES] the table's half of a stage
    uint64_t* empty = tfull + L::STAGES;                              // [STAGES]
    uint64_t* accfull = empty + L::STAGES;
    uint64_t* accempty = accfull + 1;
    uint64_t* drain = accempty + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* s_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const T* F = reinterpret_cast<const T*>(blockIdx.z ? p.F2 : p.F);
    float* out = blockIdx.z ? p.out2 : p.out;
    const long long v0 = (long long)blockIdx.x * kIV;
    const int nv = (int)min((long long)kIV, p.n_vals - v0);
    const int m0 = blockIdx.y * MT * kIM;
    if (threadIdx.x == 0) {
        for (int i = 0; i < L::STAGES; ++i) {
            mbar_init(&full[i], 4);   // the four converting warps
            mbar_init(&tfull[i], 1);  // the table's copy
            mbar_init(&empty[i], 1);
        }
        mbar_init(accfull, 1);
        mbar_init(accempty, 4 * MT);
        mbar_init(drain, 1);
        *s_abort = 0;
        mbar_fence_init();
    }
    if (threadIdx.x < kIV)
        scale[threadIdx.x] =
            (int)threadIdx.x < nv ? p.col_scale[blockIdx.z * p.n_vals + v0 + threadIdx.x] : 1.f;
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "n"(L::ALLOC)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    if (warp < 8) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kIEpiRegs));
    else asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIOtherRegs));
    bool timed_out = false;
    if (warp < 4 * MT) {
        // ---------------- accumulators -> registers ----------------
        float acc[kIV];
#pragma unroll
        for (int c = 0; c < kIV; ++c) acc[c] = 0.f;
        const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * L::ACC;
        unsigned use = 0;
        bool ok = true;
        for (int s0 = 0; s0 < n_stages; s0 += kRunStages, use ^= 1) {
            ok = warp_wait(accfull, use, s_abort, nullptr, timed_out);
            if (!ok) break;
            tc_fence_after();
            // the truncation's expected loss: a last place for a run of two or three
            // stages (measured: 0.4 a stage on spectra of random phase, 0.9 on coherent
            // ones)
            const float unb = min(kRunStages, n_stages - s0) > 1 ? 1.f + 1.1920929e-7f : 1.f;
#pragma unroll
            for (int blk = 0; blk < kIV / 8; ++blk) {
                uint32_t h[8], x[8];
                tmem_ld8(base + blk * 8, h);
                tmem_ld8(base + kIV + blk * 8, x);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    acc[blk * 8 + i] += fmaf(__uint_as_float(h[i]), unb, __uint_as_float(x[i]));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(accempty);
        }
        if (ok) {
            // scale, transpose, store: the last run's MMAs have read every stage, whose
            // memory takes the tiles
            float* tile = reinterpret_cast<float*>(smem) + warp * 32 * (kIV + 1);
#pragma unroll
            for (int c = 0; c < kIV; ++c) tile[lane * (kIV + 1) + c] = acc[c];
            __syncwarp();
            const int mw = m0 + warp * 32;
            const int rows = min(32, p.n_t - mw);
            unsigned plain[kIV / 32];  // values left to the plain sum
#pragma unroll
            for (int j = 0; j < kIV / 32; ++j) {
                const int c = lane + 32 * j;
                const float sc = c < nv ? scale[c] : 1.f;
                plain[j] = __ballot_sync(0xffffffffu, sc == 0.f);
                if (c >= nv || sc == 0.f) continue;
                const float inv = 1.f / sc;  // (2 dk follows by itself: 2 dk / sc could leave the normal range)
                float* o = out + (size_t)mw * p.n_vals + v0 + c;
#pragma unroll
                for (int r0 = 0; r0 < 32; r0 += 16) {
                    float v[16];
#pragma unroll
                    for (int r = 0; r < 16; ++r) v[r] = p.scale * (inv * tile[(r0 + r) * (kIV + 1) + c]);
                    if (p.accumulate)
#pragma unroll
                        for (int r = 0; r < 16; ++r)
                            if (r0 + r < rows) v[r] += o[(size_t)(r0 + r) * p.n_vals];
#pragma unroll
                    for (int r = 0; r < 16; ++r)
                        if (r0 + r < rows) o[(size_t)(r0 + r) * p.n_vals] = v[r];
                }
            }
            if (plain[0] | plain[1] | plain[2] | plain[3]) plain_values<T>(p, F, out, v0, nv, mw, plain);
        }
    } else if (warp == 8) {
        // ---------------- MMA issue (warp-uniform loop, one elected lane) ----------------
        const uint32_t sb = smem_u32(smem);
        bool go = true;
        unsigned run = 0;
        for (int s0 = 0; s0 < n_stages && go; s0 += kRunStages, ++run) {
            go = warp_wait(accempty, (run & 1) ^ 1, s_abort, nullptr, timed_out);
            if (!go) break;
            tc_fence_after();
            const int s1 = min(s0 + kRunStages, n_stages);
            for (int s = s0; s < s1; ++s) {
                const int st = s % L::STAGES;
                const unsigned use = (s / L::STAGES) & 1;
                go = warp_wait(&full[st], use, s_abort, nullptr, timed_out) &&
                     warp_wait(&tfull[st], use, s_abort, nullptr, timed_out);
                if (!go) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t a = sb + st * L::STAGE;
                    const uint64_t bh = smem_desc(a + MT * 2 * kAHalf, kBKStep, 128);
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        const uint64_t ah = smem_desc(a + mt * 2 * kAHalf, kAKStep, 128);
                        const uint64_t al = ah + (kAHalf >> 4);
                        const uint32_t d = tmem + mt * L::ACC;
#pragma unroll
                        for (int ks = 0; ks < 2; ++ks) {
                            const uint64_t ka = ks * (2 * kAKStep >> 4), kb = ks * (2 * kBKStep >> 4);
                            mma_f16(d, ah + ka, bh + kb, mma_idesc(kIM, 2 * kIV, false, false), s > s0 || ks > 0);
                            mma_f16(d + kIV, al + ka, bh + kb, mma_idesc(kIM, kIV, false, false), 1);
                        }
                    }
                    mma_commit(&empty[st]);
                    if (s + 1 == s1) mma_commit(accfull);
                }
                __syncwarp();
            }
        }
        // no MMA may be in flight when the tensor memory is freed
        if (elect_one()) mma_commit(drain);
        __syncwarp();
        if (mbar_wait(drain, 0) != WAIT_DONE) timed_out = true;
    } else if (warp == 9) {
        // ---------------- the phase table's stages ----------------
        if (lane == 0) {
            const unsigned char* tab = p.table + (size_t)blockIdx.y * MT * n_stages * 2 * kAHalf;
            const bool first = blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
            auto lost = [&](int s) { return first && s == p.fail_stage; };
            int issued = 0;
            for (int s = 0; s < n_stages; ++s) {
                const int st = s % L::STAGES;
                if (field_wait(&empty[st], ((s / L::STAGES) & 1) ^ 1, s_abort, nullptr, timed_out) != WAIT_DONE) break;
                // times past the table's last block of 128 have no stage: nothing reads their rows
                const int blocks = min(MT, p.m_blocks - (int)blockIdx.y * MT);
                if (lost(s)) continue;
                mbar_expect_tx(&tfull[st], blocks * 2 * kAHalf);
                for (int mt = 0; mt < blocks; ++mt)
                    bulk_g2s(smem + st * L::STAGE + mt * 2 * kAHalf, tab + ((size_t)mt * n_stages + s) * 2 * kAHalf,
                             2 * kAHalf, &tfull[st]);
                issued = s + 1;
            }
            // no copy may be on its way into this shared memory when the CTA ends:
            // wait (bounded) for the newest copy of every stage
            for (int s = max(0, issued - L::STAGES); s < issued; ++s)
                if (!lost(s) && mbar_wait(&tfull[s % L::STAGES], (s / L::STAGES) & 1) != WAIT_DONE) timed_out = true;
        }
        __syncwarp();
    } else if (warp >= 12) {
        // ---------------- the spectra's stages ----------------
        // thread = value: neighbouring lanes load neighbouring values, and the 16
        // bytes of four omegas' real and imaginary parts are one row of a K-major
        // core matrix (with values along the 16 bytes the loads touched 32 rows'
        // sectors at a time: 1.9 us a stage)
        const int c = threadIdx.x - 12 * 32;
        const float sc = scale[c];  // 0 (a value with an infinity or a NaN): zero operands
        const bool live = c < nv && sc > 0.f;
        const T* src = F + v0 + (live ? c : 0);
        // asynchronous copies several stages ahead (48 KB in flight: a stage at a
        // time in registers took 1.3 us each); every thread reads back its own
        constexpr int kAhead = kRawBytes / (kIOm * kIV * (int)sizeof(T));
        T* raw = reinterpret_cast<T*>(smem + L::OFF_RAW) + c;
        auto copy_stage = [&](int s) {
            T* dst = raw + (s % kAhead) * (kIOm * kIV);
#pragma unroll
            for (int i = 0; i < kIOm; ++i) {
                const int n = s * kIOm + i;
                const bool in = live && n < p.n_omega;
                asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_u32(dst + i * kIV)),
                             "l"(src + (in ? (size_t)n * p.n_vals : 0)), "n"((int)sizeof(T)),
                             "r"(in ? (int)sizeof(T) : 0)  // the rest is zero-filled
                             : "memory");
            }
        };
        for (int s = 0; s < kAhead - 1; ++s) {
            if (s < n_stages) copy_stage(s);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        for (int s = 0; s < n_stages; ++s) {
            const int st = s % L::STAGES;
            if (s + kAhead - 1 < n_stages) copy_stage(s + kAhead - 1);
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
            float2 f[kIOm];
#pragma unroll
            for (int i = 0; i < kIOm; ++i) {
                const float2 v = load_f32(raw + (s % kAhead) * (kIOm * kIV), i * kIV);
                f[i] = make_float2(v.x * sc, v.y * sc);
            }
            if (!warp_wait(&empty[st], ((s / L::STAGES) & 1) ^ 1, s_abort, nullptr, timed_out)) break;
            unsigned char* b = smem + st * L::STAGE + MT * 2 * kAHalf + c * 16;
#pragma unroll
            for (int k = 0; k < kIOm / 4; ++k)
                split_store8(b + k * kBKStep, b + k * kBKStep + kBKStep / 2, f + 4 * k);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[st]);
        }
        // (a stage given up on leaves copies on their way into this shared memory)
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(L::ALLOC));
    }
    if (timed_out) atomicOr(p.err, ERR_TIMEOUT);
}

template <typename T, int MT>
int launch(const IdftLaunch& p, int n_stages, cudaStream_t s)
{
    using L = Idft<MT>;
    auto kern = idft_tensor_kernel<T, MT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM);
    if (e != cudaSuccess) return -(int)e;
    const dim3 grid((unsigned)((p.n_vals + kIV - 1) / kIV), (unsigned)((p.m_blocks + MT - 1) / MT), p.F2 ? 2 : 1);
    kern<<<grid, kIThreads, L::SMEM, s>>>(p, n_stages);
    e = cudaGetLastError();
    return e == cudaSuccess ? 1 : -(int)e;
}

}  // namespace

// A tile of 128 values costs about 17 us before its first product (start,
// tensor memory, stores), which the FP32 kernel's tiles of 64 x 64 do not pay:
// 16384 points, 64 times: 48 omegas 65 us there, 74 here; 256 and 200 times: 824
// against 189; 16 omegas and 1000 times: 237 against 227, 8: 147 against 224.
bool idft_on_tensor(int n_omega, int n_t)
{
    return n_omega >= 16 && (long long)n_omega * ((n_t + 63) / 64) >= 96;
}

size_t idft_scratch_bytes(int n_omega, long long n_vals, int n_t)
{
    return (size_t)((n_t + kIM - 1) / kIM) * ((n_omega + kIOm - 1) / kIOm) * 2 * kAHalf + 2 * n_vals * sizeof(float);
}

int launch_idft_tensor(const IdftLaunch& in, cudaStream_t s)
{
    IdftLaunch p = in;
    p.scale = (float)(2.0 * p.dk);
    p.m_blocks = (p.n_t + kIM - 1) / kIM;
    const int n_stages = (p.n_omega + kIOm - 1) / kIOm, n_table = p.m_blocks * n_stages;
    p.col_scale = reinterpret_cast<float*>(p.table + (size_t)n_table * 2 * kAHalf);
    const unsigned blocks = (unsigned)(n_table + (p.F2 ? 2 : 1) * ((p.n_vals + kScanCols - 1) / kScanCols));
    if (p.f64) idft_prep_kernel<double2><<<blocks, kIM, 0, s>>>(p, n_stages, n_table);
    else idft_prep_kernel<float2><<<blocks, kIM, 0, s>>>(p, n_stages, n_table);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return -(int)e;
    int r;
    if (p.m_blocks == 1)
        r = p.f64 ? launch<double2, 1>(p, n_stages, s) : launch<float2, 1>(p, n_stages, s);
    else
        r = p.f64 ? launch<double2, 2>(p, n_stages, s) : launch<float2, 2>(p, n_stages, s);
    return r < 0 ? r : 1 + r;
}

}  // namespace sc
