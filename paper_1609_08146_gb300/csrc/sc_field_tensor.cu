// sc_field_tensor.cu -- the FP32 field sum as a contraction on the tensor
// cores (tcgen05), for chunks of a few dozen to 256 omegas.  The quadrature of
// Sec. II, Eq. 11 over the node table with the compensated phase of
// Sec. III.C.1; see sc_field.cu for the summand.
//
// For one point the sums over the nodes j are S_c(omega) = sum_j C_cj e^{i k
// Phi_j} with twelve real coefficients per pair,
//     C = (U + V, Wv, V/R, Wv/R),  E = ik S_{U+V} - S_{V/R},  B = ik S_W - S_{W/R}.
// On the uniform grid omega = Omega_{n1} + delta_{n2} the phase factor is a
// product of a row phasor e^{i 2 pi Omega_{n1} Phi} and a column phase
// theta_{n2} = 2 pi delta_{n2} Phi, with the offsets delta symmetric about
// zero, so that +delta and -delta share their cosine and sine columns:
//     D[row, col] = sum_j A[row, j] B[col, j]
//   rows  R row phasors, cosine and sine (M = 2 R = 64 or 128),
//   cols  12 coefficients times N2 trigonometric columns (N = 12 N2),
//   K     the nodes.
// N2 omegas per row phasor come out of 12 N2 real columns: no product is
// computed twice, and a pair costs 2 R + 12 N2 operand values instead of the
// direct kernel's 24 FP32 operations for each of its R N2 omegas.
//
// Precision.  Every operand value x is split into two halves, hi = fp16(x) and
// lo = fp16(x - hi), 22 bits in all, and three products are accumulated: hi hi
// in one set of TMEM columns, hi lo + lo hi in another.  What is dropped (lo
// lo and the rounding of lo) is below 2^-23 of the largest operand, the size
// of one FP32 rounding.  The coefficients are brought into the range of fp16
// by powers of two chosen per point from bounds on the table's largest source
// and the smallest distance.  The tensor cores' accumulation drops the bits
// below the accumulator's last place instead of rounding, which makes coherent
// sums too small, by half a last place per MMA (measured: 1.2e-7 per node
// tile).  So a run of accumulation is only kFoldTiles tiles (160 nodes; the
// direct kernel's FP32 runs have 2048), the expected loss, one last place per
// tile after the first, is given back when the run is read, and the runs are
// summed outside the tensor cores by Kahan's rule.  Against FP64, relative
// norms over sizes and beams at random: 1.9e-7 to 4.1e-7 here, 2.8e-7 to
// 1.1e-6 with the FP32 kernels.
//
// What bounds it.  256 omegas, 512^2 nodes, 4160 points: 51.7 ms, 5.4e12
// evaluations a second (direct kernel, at 0.84 of the FP32 pipe: 232 ms).
// Shared memory is busy 91% of the time (54% by the LSU, mostly the operands'
// stores, 38% by the MMAs' reads of them); the schedulers issue in 64% of the
// cycles, and the tensor pipe works 31%.  At a few dozen omegas a tile's fixed work (the
// pair's geometry, three rotations, barriers) counts for most of it: at 48 omegas
// shared memory is busy 75% and the schedulers issue in 68% of the cycles, at 100
// omegas 86% and 67%.  No one of them binds alone there: twenty stages (a producer
// then need not wait) and the halves of A stacked into one M = 128 MMA (fewer MMAs
// and reads) each gained nothing.
//
// Where the lines between the classes lie (256^2 nodes, 4160 points, 1e11
// evaluations a second): 24 omegas, direct 9.8, here 8.5; 25: 8.3 and 10.8; 48:
// 10.4 and 17.8.  32 row phasors of 2 omegas up to 64 omegas (25: 10.5 against 9.5
// with 64 rows, whose reads of shared memory M = 64 halves; 64: 21.1 against 21.5),
// of 4 up to 128 (128: 33.9 against 30.7 on 64 rows of 2, with a quarter fewer
// operand values; 100: 26.5, 25.5), 64 rows of 4 above (256: 52.1; rows of 3 from
// 129 to 192 are no better: 160: 37.3 against 39.6, 192: 42.3 against 44.5).
//
// Structure (one CTA per SM, 16 warps; shared memory holds ten stages):
//   warps 0-3   read a finished accumulator (TMEM, two or four), keep the
//               compensated running sums of the item (one point, one node
//               split) in registers and write its partials;
//   warps 4, 8  issue the MMAs, a warp for every second run;
//   the others  produce operands, each into a stage of its own: lane = node,
//               five warps for every second run.  A lane computes its pair's
//               geometry, coefficients and phases and writes its operand
//               columns in the MN-major core-matrix layout (8 rows of one node
//               are 16 contiguous bytes, so that a warp's stores are
//               conflict-free); no data passes between lanes.
// Items are strided over the CTAs (item = blockIdx + i gridDim), which every
// role follows on its own; all waits are bounded as in the other kernels, and of a
// whole warp.  Items whose points do not qualify for fp16 operands come last, on all
// sixteen warps (plain_items).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sc_field_common.cuh"
#include "sc_internal.h"
#include "sc_tensor.cuh"

namespace sc {

namespace {

constexpr int kFoldTiles = 5;               // node tiles per run of an accumulator
constexpr int kStages = 2 * kFoldTiles;     // operand stages (one node tile each): half for either accumulator
constexpr int kProd = kStages;              // producer warps, each with a stage of its own
constexpr int kTensorThreads = 512, kWarps = kTensorThreads / 32;
static_assert(4 + 2 + kProd <= kTensorThreads / 32, "warps");
// Registers: 128 a thread at launch; the epilogue's warpgroup takes 176 and
// the other three 112 (128 * 176 + 384 * 112 = 65536).
constexpr int kLaunchRegs = 128, kEpiRegs = 176, kOtherRegs = 112;
static_assert(128 * kEpiRegs + 384 * kOtherRegs <= 512 * kLaunchRegs, "register split");
constexpr int kBlkBytes = kTile * 16;           // a block of 8 rows (or columns) of a stage's 32 nodes

// N2 omegas per row phasor, R row phasors (M = 2 R rows of A)
template <int N2, int R>
struct Tens {
    static constexpr int ABYTES = 2 * R / 8 * kBlkBytes;  // one half (hi or lo) of A
    static constexpr int N = 12 * N2;
    static constexpr int DCOLS = 2 * N;            // one accumulator: hi hi, then hi lo + lo hi
    // Accumulators in tensor memory: with four the MMAs need not wait for the
    // epilogue's last read (25 omegas 6.41 -> 6.23 ms, 64 8.17 -> 7.99); more columns
    // gain nothing at 256 omegas and cost 2% on small tables.
    static constexpr int ACCS = N2 <= 2 ? 4 : 2;
    static constexpr int ALLOC = ACCS * DCOLS <= 64 ? 64 : (ACCS * DCOLS <= 128 ? 128 : (ACCS * DCOLS <= 256 ? 256 : 512));
    static constexpr int STAGE = 2 * ABYTES + 2 * (N / 8) * kBlkBytes;
    static constexpr int OFF_BAR = kStages * STAGE;
    static constexpr int SMEM = OFF_BAR + 256;
    static_assert(N2 % 2 == 0 && N % (R == 64 ? 16 : 8) == 0, "column pairs, product widths (M = 128 wants 16s)");
    static_assert(ACCS * DCOLS <= ALLOC, "tensor memory");
    static_assert(SMEM <= 227 * 1024, "shared memory");
    // a warp's share of the stages in plain_item(): its sums, or its pair rows
    static_assert(OFF_BAR / kWarps / 16 * 16 >= R * N2 * kAcc * 4 && OFF_BAR / kWarps / 16 * 16 >= (32 * 16 + 8 * 4) * 4,
                  "plain loop");
};

// Stage layout, MN-major: 128 bytes from one block of 8 nodes to the next,
// kBlkBytes from one block of 8 rows or columns to the next.
__device__ __forceinline__ uint64_t stage_desc(uint32_t addr) { return smem_desc(addr, 128, kBlkBytes); }

// Segments of eight row phasors that n_omega omegas take, and the one the
// seeds start from (then outwards both ways).
__host__ __device__ inline int segments(int n_omega, int n2) { return ((n_omega + n2 - 1) / n2 + 7) / 8; }
__host__ __device__ inline int seed_seg(int nseg) { return nseg >> 1; }

// ------------------------------------------------------------------------
// One work item as every role sees it.

struct TItem {
    const FieldLaunch* f;
    int pt, split, t0, nt;
    float4 P;        // point and |r'|^2
    float js, rs;    // powers of two: sources times js, 1/R times rs
    bool ok;         // operands fit fp16 (see below); otherwise the item takes the plain FP32 loop
};

__device__ __forceinline__ TItem tensor_item(const BatchLaunch& b, long long item)
{
    // decode(), with a 32-bit division where it can be (every role of every
    // item pays for it; the 64-bit one takes over a hundred instructions)
    Item w;
    w.r = find_req(b, item);
    const long long local = item - w.r->item0;
    if (local >> 32) {
        w = decode(b, item);
    } else {
        w.split = (int)((unsigned)local / (unsigned)w.r->pb);
        w.pbi = (int)((unsigned)local % (unsigned)w.r->pb);
    }
    TItem t;
    t.f = &w.r->f;
    t.pt = w.pbi;
    t.split = w.split;
    int t1;
    split_range(*t.f, w.split, t.t0, t1);
    t.nt = t1 - t.t0;
    load_point(t.f->pts, t.f->n_pts, w.pbi, t.P);  // (|r'|^2 dropped by the roles that do not use it)
    // R >= |P| - |r'| >= rmin on every node; |J|, |rho| <= amax.  The powers of
    // two bring |U + V|, |Wv| below 2^12 and 1/R below 1.  Points within 1/16
    // of the mirror's smallest distance (or sources out of range, or NaN) do
    // not qualify: their 1/R spans too much for one scale.
    const float amax = w.split < t.f->n_splits ? t.f->amax_surf : t.f->amax_rim;
    const float rmin = t.f->pmin - sqrtf(fmaf(t.P.x, t.P.x, fmaf(t.P.y, t.P.y, t.P.z * t.P.z)));
    t.ok = rmin >= 0.0625f * t.f->pmin && rmin > 1e-30f && rmin < 1e30f && amax < 1e30f && amax >= 0.f;
    t.js = t.rs = 1.f;
    if (t.ok) {
        t.rs = ldexpf(1.f, ilogbf(rmin));
        if (amax > 0.f) {
            const int e = 10 - ilogbf(amax / rmin);
            t.ok = e > -100 && e < 100;
            t.js = t.ok ? ldexpf(1.f, e) : 1.f;
        }
    }
    return t;
}

// The launch's abort word, read between items by the MMA warps, which pass it
// on to their CTA's word; every wait of the other roles ends on that.
__device__ __forceinline__ bool launch_aborted(const BatchLaunch& b, volatile int* s_abort)
{
    if (b.abort && *(const volatile int*)b.abort) *s_abort = 1;
    return *s_abort != 0;
}

// ------------------------------------------------------------------------
// Producers

// One segment: eight row phasors from the seed of its fourth, its neighbour by
// one rotation, and the three-term recurrence from these two outwards: three
// steps at most, so that the rounding of c = 2 cos, which n steps multiply by
// n (n + 1) / 2, is multiplied by 6 and not by the 21 of a chain from one end.
// Steps alternate -c, -c, +c, which saves the negation; slots 1, 2, 5, 6 come
// out negated and the epilogue turns them back.
template <int ABYTES>
__device__ __forceinline__ void store_segment(unsigned char* a_hi, float2 seed, float2 rot, float2 cc, float2 ncc)
{
    float2 ph[8];
    ph[3] = seed;
    ph[4] = cmul(seed, rot);
#pragma unroll
    for (int j = 1; j < 4; ++j) {
        ph[4 + j] = __ffma2_rn((j & 1) ? ncc : cc, ph[3 + j], ph[2 + j]);
        ph[3 - j] = __ffma2_rn((j & 1) ? ncc : cc, ph[4 - j], ph[5 - j]);
    }
    const float2 c[4] = {make_float2(ph[0].x, ph[1].x), make_float2(ph[2].x, ph[3].x),
                         make_float2(ph[4].x, ph[5].x), make_float2(ph[6].x, ph[7].x)};
    const float2 d[4] = {make_float2(ph[0].y, ph[1].y), make_float2(ph[2].y, ph[3].y),
                         make_float2(ph[4].y, ph[5].y), make_float2(ph[6].y, ph[7].y)};
    split_store8(a_hi, a_hi + ABYTES, c);
    split_store8(a_hi + kBlkBytes, a_hi + ABYTES + kBlkBytes, d);
}

// One tile's operands; `wait` (bounded) blocks until the MMAs have read the
// stage's last contents and is placed after everything that can be computed
// without the stage.  False: aborted or expired.
template <int N2, int R, typename Wait>
__device__ __forceinline__ bool produce_tile(unsigned char* stage, const float nd[9], const TItem& it, int lane,
                                             int nseg, const TensorSteps& w, Wait wait)
{
    using L = Tens<N2, R>;
    const float px = nd[0], py = nd[1], pz = nd[2], pn = nd[3], wo = nd[4];
    const float4 P = it.P;
    // pair geometry and phase as in pair_coefs()
    const float dx = px - P.x, dy = py - P.y, dz = pz - P.z;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float ir = rsqrtf(r2);
    const float dist = r2 * ir;
    const float D = fmaf(-2.0f * P.x, px, fmaf(-2.0f * P.y, py, fmaf(-2.0f * P.z, pz, P.w)));
    const float phi = __fdividef(D, dist + pn) + wo;
    const float rx = dx * ir, ry = dy * ir, rz = dz * ir;
    const float sir = it.js * ir;
    const float ux = nd[5] * sir, uy = nd[6] * sir, uz = nd[7] * sir;
    const float a = nd[8] * sir;
    const float irs = ir * it.rs;
    float co[12];
    const float vx = a * rx, vy = a * ry, vz = a * rz;
    co[0] = ux + vx; co[1] = uy + vy; co[2] = uz + vz;
    co[3] = fmaf(uy, rz, -uz * ry);
    co[4] = fmaf(uz, rx, -ux * rz);
    co[5] = fmaf(ux, ry, -uy * rx);
    co[6] = vx * irs; co[7] = vy * irs; co[8] = vz * irs;
    co[9] = co[3] * irs; co[10] = co[4] * irs; co[11] = co[5] * irs;

    // cosines and sines of the column offsets, m + 1/2 steps
    float trig[N2];
    {
        float2 q = rotation_2wphi(w.col.x, w.col.y, phi);
        const float2 full = cmul(q, q);
#pragma unroll
        for (int m = 0; m < N2 / 2; ++m) {
            trig[2 * m] = q.x;
            trig[2 * m + 1] = q.y;
            if (m + 1 < N2 / 2) q = cmul(q, full);
        }
    }
    // row phasors: one seed (MUFU sine and cosine, as in the direct kernel) and
    // the rotations between rows and between segments
    const float2 rot = rotation_2wphi(w.row.x, w.row.y, phi);
    const float2 rseg = rotation_2wphi(w.seg.x, w.seg.y, phi);
    float2 up = phasor_2wphi_mufu(w.seed.x, w.seed.y, phi);
    if (!wait()) return false;

    unsigned char* b_hi = stage + 2 * L::ABYTES + lane * 16;
    unsigned char* b_lo = b_hi + (L::N / 8) * kBlkBytes;
#pragma unroll
    for (int blk = 0; blk < L::N / 8; ++blk) {
        float2 v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c0 = blk * 8 + 2 * i;
            v[i].x = co[c0 % 12] * trig[c0 / 12];
            v[i].y = co[(c0 + 1) % 12] * trig[(c0 + 1) / 12];
        }
        split_store8(b_hi + blk * kBlkBytes, b_lo + blk * kBlkBytes, v);
    }
    // segments outwards from the seed's, two independent chains
    const float2 cc = make_float2(2.f * rot.x, 2.f * rot.x);
    const float2 ncc = make_float2(-cc.x, -cc.y);
    const float2 rback = make_float2(rseg.x, -rseg.y);
    float2 dn = cmul(up, rback);
    const int s0 = seed_seg(nseg);
    unsigned char* a_up = stage + lane * 16 + 2 * s0 * kBlkBytes;
    unsigned char* a_dn = a_up - 2 * kBlkBytes;
    store_segment<L::ABYTES>(a_up, up, rot, cc, ncc);
    const int both = nseg - 1 - s0;  // segments on either side (an even count has one more below)
#pragma unroll 1
    for (int s = 0; s < both; ++s) {
        up = cmul(up, rseg);
        a_up += 2 * kBlkBytes;
        store_segment<L::ABYTES>(a_dn, dn, rot, cc, ncc);
        store_segment<L::ABYTES>(a_up, up, rot, cc, ncc);
        a_dn -= 2 * kBlkBytes;
        dn = cmul(dn, rback);
    }
    if (s0 > both) store_segment<L::ABYTES>(a_dn, dn, rot, cc, ncc);
    return true;
}

__device__ __forceinline__ void load_node(const FieldLaunch& p, int tile, int lane, float nd[9])
{
    const float* src = p.nodes + (size_t)tile * kTileFloats + lane;
#pragma unroll
    for (int f = 0; f < 9; ++f) nd[f] = __ldg(src + f * kTile);
}

// ------------------------------------------------------------------------
// Epilogue

__device__ __forceinline__ void two_sum(float& s, float& e, float v)
{
    const float t = s + v, b = t - s;
    e += (s - (t - b)) + (v - b);
    s = t;
}

// The item's partials from the running sums s - e of the lane's row.  With CC,
// CS the cosine row's sums over the cosine and sine columns of an offset
// phi > 0, and SC, SS the sine row's, the sums at +-phi are
//     Re = CC -+ SS,   Im = SC +- CS,
// and E = ik S1 - S2, B likewise (S1 over U + V or Wv, S2 over V/R or Wv/R).  A
// cosine row (lane) writes real parts, Re E = -k Im S1 - Re S2, its partner (lane
// ^ 8) imaginary ones, Im E = k Re S1 - Im S2: either needs the partner's cosine
// column of S1 and sine column of S2, one exchange each.
template <int N2>
__device__ __forceinline__ void write_item(const TItem& it, int row, bool own_row, const float2* s2,
                                           const float2* e2)
{
    const FieldLaunch& p = *it.f;
    const int seg = row >> 4, idx = row & 7;
    const bool im = (row & 8) != 0;
    const int n1 = seg * 8 + idx;
    const float sg = ((idx + 1) & 2) ? -1.f : 1.f;
    const float inv = sg / it.js, inv2 = 1.0f / it.rs;
    auto s = [&](int c) { return (c & 1) ? s2[c >> 1].y : s2[c >> 1].x; };
    auto e = [&](int c) { return -((c & 1) ? e2[c >> 1].y : e2[c >> 1].x); };
    float2* base = p.ws + (((size_t)it.split * p.n_pts + it.pt) * (size_t)p.n_omega) * kAcc + (im ? 1 : 0);
#pragma unroll
    for (int o = 0; o < N2 / 2; ++o) {  // offsets, pairs +-phi
        const int tc = 2 * o;  // its cosine column
        float2 dst_v[2][6];
        float k_h[2], k_l[2];
        int nn[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // h = 0: +phi, 1: -phi
            const int twice = (h == 0 ? 1 : -1) * (2 * o + 1);
            nn[h] = n1 * N2 + (twice + N2 - 1) / 2;
            // k_n = k_0 + n dk as a float-float pair, with the sign of ik's product
            const float fn = (float)nn[h], a = fn * p.steps.dk.x;
            float kh = p.steps.k0.x, kl = fmaf(fn, p.steps.dk.x, -a) + fmaf(fn, p.steps.dk.y, p.steps.k0.y);
            two_sum(kh, kl, a);
            k_h[h] = im ? kh : -kh;
            k_l[h] = im ? kl : -kl;
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const int c1 = tc * 12 + c, c2 = c1 + 6;
            // partner's cosine column of S1 and sine column of S2
            const float p1 = __shfl_xor_sync(0xffffffffu, s(c1), 8), p1e = __shfl_xor_sync(0xffffffffu, e(c1), 8);
            const float p2 = __shfl_xor_sync(0xffffffffu, s(c2 + 12), 8);
            const float p2e = __shfl_xor_sync(0xffffffffu, e(c2 + 12), 8);
            const float o1 = s(c1 + 12), o1e = e(c1 + 12);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float q1 = (im ? -1.f : 1.f) * (h == 0 ? 1.f : -1.f);  // S1: cosine rows +-, sine rows -+
                const float q2 = -q1;                                       // S2: cosine rows -+, sine rows +-
                float a = p1, al = fmaf(q1, o1e, p1e);
                two_sum(a, al, q1 * o1);
                float v = k_h[h] * a;
                float vl = fmaf(k_h[h], a, -v) + fmaf(k_h[h], al, k_l[h] * a);
                float r = s(c2), rl = fmaf(q2, p2e, e(c2));
                two_sum(r, rl, q2 * p2);
                two_sum(v, vl, -r * inv2);
                dst_v[h][c] = make_float2(inv * v, inv * fmaf(-rl, inv2, vl));
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (own_row && nn[h] < p.n_omega)
#pragma unroll
                for (int c = 0; c < 6; ++c) base[(size_t)nn[h] * kAcc + 2 * c] = dst_v[h][c];
    }
}

// ------------------------------------------------------------------------
// Items whose operands do not fit fp16 (points near the mirror or beyond it): the
// direct kernel's loop, on all sixteen warps once the tile loop is done and the
// registers are shared out evenly again.  A warp sums every sixteenth node tile: GP
// lanes of NB consecutive omegas share a node, 32 / GP nodes side by side, from
// pair rows in the warp's part of the stages.  Every flush the node groups' sums
// are added within the warp, then the warps' in warp order to the compensated
// partials.
//
// What bounds it: the FP32 pipe, as in the direct kernel, whose rate it keeps (all
// points off the focus, 128^2 nodes, 2048 points, this against the direct kernel: 25
// omegas 1.14 ms and 1.18, 64 2.19 and 2.20, 128 3.99 and 3.92, 256 7.73 and 7.68;
// ten producer warps with their 112 registers and a seed for every two omegas
// took 3.33, 3.35, 5.36 and 18.9).  On tables of a few tiles a warp an item's start
// shows (32^2 nodes, 512 points: 25 omegas 67 us and 133, 128 158 and 142).

// lanes per node and omegas per lane, as in the direct kernel's classes from 25 omegas on
__device__ __forceinline__ int plain_lanes(int n_omega)
{
    return n_omega <= 32 ? 4 : (n_omega <= 64 ? 8 : (n_omega <= 128 ? 16 : 32));
}

// w + n d as a float-float pair
__device__ __forceinline__ float2 ff_step(float2 w, float n, float2 d)
{
    const float a = n * d.x;
    float h = w.x, l = fmaf(n, d.x, -a) + fmaf(n, d.y, w.y);
    two_sum(h, l, a);
    return make_float2(h, l);
}

// Halve the slots a lane keeps: lanes that differ in `bit` exchange what the other
// keeps and add.
template <int KEEP>
__device__ __forceinline__ void halve(AccX2* v, int lane, int bit)
{
    const bool up = (lane & bit) != 0;
#pragma unroll
    for (int j = 0; j < KEEP; ++j)
#pragma unroll
        for (int c = 0; c < kAcc / 2; ++c) {
            const float2 lo = v[j].v[c], hi = v[j + KEEP].v[c];
            const float2 give = up ? lo : hi, keep = up ? hi : lo;
            v[j].v[c].x = keep.x + __shfl_xor_sync(0xffffffffu, give.x, bit);
            v[j].v[c].y = keep.y + __shfl_xor_sync(0xffffffffu, give.y, bit);
        }
}

template <int NB>
__device__ __forceinline__ void plain_item(unsigned char* smem, int warp_bytes, const FieldLaunch& p, float4 P, int pt,
                                        int split, int t0, int nt)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gp = plain_lanes(p.n_omega), g = lane & (gp - 1);
    float* mine = reinterpret_cast<float*>(smem + warp * warp_bytes);
    float* row0 = mine + (lane & ~(gp - 1)) * 16 + lane / gp * 4;  // the lane's nodes (4 floats of pad: banks)
    const float2 w = ff_step(make_float2(p.om_hi0, p.om_lo0), (float)(g * NB), make_float2(p.dom_hi, p.dom_lo));
    float kv[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        const float2 k = ff_step(p.steps.k0, (float)(g * NB + j), p.steps.dk);
        kv[j] = k.x + k.y;
    }
    float2* dst = p.ws + ((size_t)split * p.n_pts + pt) * (size_t)p.n_omega * kAcc;
    const int round = min(max(1, p.flush_tiles), 1 << 20) * kWarps;  // tiles per flush, all warps
    // fewer tiles than warps (a rim, a small table): `share` warps take a tile's nodes
    int share = 1;
    while (2 * share * nt <= kWarps && 2 * share <= gp) share *= 2;
    const int q0 = warp % share * (gp / share), q1 = q0 + gp / share;
    for (int r0 = 0; r0 < nt || r0 == 0; r0 += round) {
        AccX2 acc[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int c = 0; c < kAcc / 2; ++c) acc[j].v[c] = make_float2(0.f, 0.f);
        for (int t = r0 + warp / share; t < min(nt, r0 + round); t += kWarps / share) {
            const float* nb = p.nodes + (size_t)(t0 + t) * kTileFloats;
            float co[10];
            const float phi = pair_coefs(nb, lane, P, co);
            const float2 rot = phasor_2wphi(p.dom_hi, p.dom_lo, phi);
            float4* r4 = reinterpret_cast<float4*>(mine + lane * 16 + lane / gp * 4);
            r4[0] = make_float4(co[0], co[1], co[2], co[3]);
            r4[1] = make_float4(co[4], co[5], co[6], co[7]);
            r4[2] = make_float4(co[8], co[9], rot.x, rot.y);
            r4[3] = make_float4(phi, 0.f, 0.f, 0.f);
            __syncwarp();
#pragma unroll 1
            for (int q = q0; q < q1; ++q) {
                const float4* s4 = reinterpret_cast<const float4*>(row0 + q * 16);
                const float4 a0 = s4[0], a1 = s4[1], a2 = s4[2];
                const float2 cp[10] = {make_float2(a0.x, a0.x), make_float2(a0.y, a0.y), make_float2(a0.z, a0.z),
                                       make_float2(a0.w, a0.w), make_float2(a1.x, a1.x), make_float2(a1.y, a1.y),
                                       make_float2(a1.z, a1.z), make_float2(a1.w, a1.w), make_float2(a2.x, a2.x),
                                       make_float2(-a2.y, -a2.y)};
                const float2 ro = make_float2(a2.z, a2.w);
                const float2 cc = make_float2(2.f * ro.x, 2.f * ro.x), ncc = make_float2(-cc.x, -cc.x);
                float2 p0 = phasor_2wphi_mufu(w.x, w.y, s4[3].x);
                float2 p1 = cmul(p0, ro);
                eval_x2<true>(acc[0], cp, kv[0], p0);
                eval_x2<true>(acc[1], cp, kv[1], p1);
#pragma unroll
                for (int j = 2; j < NB; ++j) {
                    const float2 pn = __ffma2_rn((j & 1) ? cc : ncc, p1, p0);
                    eval_x2<true>(acc[j], cp, kv[j], pn);
                    p0 = p1;
                    p1 = pn;
                }
            }
            __syncwarp();
        }
        // the node groups' sums: every lane ends with 8 gp / 32 of its omegas
        int slot0 = 0, slots = 8;
        if (gp <= 16) halve<4>(acc, lane, 16), slots = 4, slot0 += (lane & 16) >> 2;
        if (gp <= 8) halve<2>(acc, lane, 8), slots = 2, slot0 += (lane & 8) >> 2;
        if (gp <= 4) halve<1>(acc, lane, 4), slots = 1, slot0 += (lane & 4) >> 2;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int slot = slot0 + j;
            if (j < slots && slot < NB) {
                const float sg = (slot & 2) ? -1.f : 1.f;  // sign carried by the phasor recurrence
                float4* r4 = reinterpret_cast<float4*>(mine + (g * NB + slot) * kAcc);
#pragma unroll
                for (int c = 0; c < kAcc / 4; ++c)
                    r4[c] = make_float4(sg * acc[j].v[2 * c].x, sg * acc[j].v[2 * c].y, sg * acc[j].v[2 * c + 1].x,
                                        sg * acc[j].v[2 * c + 1].y);
            }
        }
        __syncthreads();
        for (int x = threadIdx.x; x < p.n_omega * kAcc; x += kTensorThreads) {
            float2 v = r0 == 0 ? make_float2(0.f, 0.f) : dst[x];
            for (int u = 0; u < kWarps; ++u) two_sum(v.x, v.y, reinterpret_cast<const float*>(smem + u * warp_bytes)[x]);
            dst[x] = v;
        }
        __syncthreads();
    }
}

// Every item of the CTA that is left to the plain loop.  Inlined at the kernel's end:
// as a call it slowed the tile loop, whose registers the compiler then divides
// differently (48 omegas, 256^2 nodes, 4096 points: 7.37 ms, 7.13 inlined).
__device__ __forceinline__ void plain_items(const BatchLaunch& b, unsigned char* smem, int bytes)
{
    const int wb = bytes / kWarps / 16 * 16;
    for (long long item = blockIdx.x; item < b.n_items; item += gridDim.x) {
        const TItem it = tensor_item(b, item);
        if (it.ok) continue;
        const int lanes = plain_lanes(it.f->n_omega);
        switch ((it.f->n_omega + lanes - 1) / lanes) {
        case 5: plain_item<5>(smem, wb, *it.f, it.P, it.pt, it.split, it.t0, it.nt); break;
        case 6: plain_item<6>(smem, wb, *it.f, it.P, it.pt, it.split, it.t0, it.nt); break;
        case 7: plain_item<7>(smem, wb, *it.f, it.P, it.pt, it.split, it.t0, it.nt); break;
        default: plain_item<8>(smem, wb, *it.f, it.P, it.pt, it.split, it.t0, it.nt);
        }
    }
}

// ------------------------------------------------------------------------

// Producer number of a warp that is neither epilogue nor MMA (4, 8): first the
// warps of the three schedulers without MMA warps (warp mod 4 = 1, 2, 3).
__device__ __forceinline__ int prod_index(int warp)
{
    return (warp & 3) ? 3 * ((warp >> 2) - 1) + (warp & 3) - 1 : 9;
}

template <int N2, int R>
__global__ void __launch_bounds__(kTensorThreads, 1) field_tensor_kernel(const __grid_constant__ BatchLaunch b)
{
    using L = Tens<N2, R>;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR);  // [kStages] stage written
    uint64_t* empty = full + kStages;                                 // [kStages] stage read by the MMAs
    uint64_t* accfull = empty + kStages;                              // [ACCS] accumulator finished
    uint64_t* accempty = accfull + L::ACCS;                           // [ACCS] accumulator read
    uint64_t* drain = accempty + L::ACCS;                             // [2] the MMA warps' last commits
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 2);
    volatile int* s_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* s_plain = s_abort + 1;                              // some item is left to the plain loop
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < L::ACCS; ++i) {
            mbar_init(&accfull[i], 1);
            mbar_init(&accempty[i], 4);
        }
        mbar_init(&drain[0], 1);
        mbar_init(&drain[1], 1);
        *s_abort = 0;
        *s_plain = 0;
        mbar_fence_init();
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "n"(L::ALLOC)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    bool timed_out = false;

    if (warp < 4) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
    else asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
    if (warp < 4) {
        // ---------------- epilogue ----------------
        // M = 128: lane = row; M = 64: 16 rows in the first half of every warp's lanes
        const int row = R == 64 ? warp * 32 + lane : warp * 16 + (lane & 15);
        const bool own_row = R == 64 || lane < 16;
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        long long fb = 0;
        bool stop = false;
        for (long long item = blockIdx.x; item < b.n_items && !stop; item += gridDim.x) {
            if (warp_aborted(s_abort)) break;
            const TItem it = tensor_item(b, item);
            if (!it.ok) {
                *s_plain = 1;
                continue;
            }
            const int ft = min(kFoldTiles, it.f->flush_tiles);
            float2 s[L::N / 2], e[L::N / 2];
#pragma unroll
            for (int c = 0; c < L::N / 2; ++c) s[c] = e[c] = make_float2(0.f, 0.f);
            const float2 neg = make_float2(-1.f, -1.f);
            for (int t = 0; t < it.nt; t += ft, ++fb) {
                const int buf = (int)(fb % L::ACCS);
                if (!warp_wait(&accfull[buf], (unsigned)((fb / L::ACCS) & 1), s_abort, b.abort, timed_out)) {
                    stop = true;
                    break;
                }
                tc_fence_after();
                const float ub = 1.f + 1.1920929e-7f * (float)(min(ft, it.nt - t) - 1);  // see Precision above
                const float2 unb = make_float2(ub, ub);
                const uint32_t base = lane_base + buf * L::DCOLS;
#pragma unroll
                for (int blk = 0; blk < L::N / 8; ++blk) {
                    uint32_t h[8], x[8];
                    tmem_ld8(base + blk * 8, h);
                    tmem_ld8(base + L::N + blk * 8, x);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int c = blk * 4 + i;
                        if (c < L::N / 2) {
                            const float2 v = __ffma2_rn(
                                make_float2(__uint_as_float(h[2 * i]), __uint_as_float(h[2 * i + 1])), unb,
                                make_float2(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1])));
                            // Kahan: the running sum is s - e
                            const float2 y = __ffma2_rn(e[c], neg, v);
                            const float2 u = __fadd2_rn(s[c], y);
                            e[c] = __ffma2_rn(y, neg, __ffma2_rn(s[c], neg, u));
                            s[c] = u;
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&accempty[buf]);
            }
            if (!stop) write_item<N2>(it, row, own_row, s, e);
        }
    } else if (warp == 4 || warp == 8) {
        // ---------------- MMA issue ----------------
        // The whole warp runs the loop and every condition and loaded value is
        // made warp-uniform by a vote or a broadcast, so that descriptors and
        // addresses live in uniform registers, where the MMA takes them from;
        // one elected lane issues.  Issued from a one-lane branch each MMA cost
        // about 200 cycles.  Two warps, taking turns by runs: a tile's barrier,
        // four MMAs and commit take one warp over 400 cycles, most of them
        // latency, and the producers make a tile in 440.
        const unsigned mine = warp == 8;
        constexpr unsigned kAll = 0xffffffffu;
        const uint64_t ah0 = stage_desc(smem_u32(smem));
        const bool leader = elect_one();
        unsigned fb = 0;  // run number: warp and stages fb & 1, accumulator fb % ACCS
        bool go = true;
        for (long long item = blockIdx.x; item < b.n_items && go; item += gridDim.x) {
            if (__any_sync(kAll, launch_aborted(b, s_abort))) break;
            const TItem it = tensor_item(b, item);
            const int nt = __shfl_sync(kAll, it.ok ? it.nt : 0, 0);
            const int ft = __shfl_sync(kAll, min(kFoldTiles, it.f->flush_tiles), 0);
            for (int t = 0; t < nt && go; t += ft, ++fb) {
                if ((fb & 1) != mine) continue;
                const unsigned buf = fb % L::ACCS, use = (fb >> 1) & 1;
                // the accumulator's last run has been read (the first waits pass at once)
                go = warp_wait(&accempty[buf], ((fb / L::ACCS) & 1) ^ 1, s_abort, b.abort, timed_out);
                if (!go) break;
                tc_fence_after();
                const uint32_t d = tmem + buf * L::DCOLS;
                const uint64_t ab = ah0 + mine * (kFoldTiles * (L::STAGE >> 4));
                uint64_t* fullb = full + mine * kFoldTiles;
                uint64_t* emptyb = empty + mine * kFoldTiles;
                const int cnt = min(ft, nt - t);
                bool ready = mbar_test(&fullb[0], use);
#pragma unroll
                for (int i = 0; i < kFoldTiles; ++i) {
                    if (!__all_sync(kAll, ready))
                        go = warp_wait(&fullb[i], use, s_abort, b.abort, timed_out);
                    if (!go) break;
                    if (i + 1 < kFoldTiles) ready = mbar_test(&fullb[i + 1], use);  // asked for ahead
                    const uint64_t ah = ab + i * (L::STAGE >> 4);
                    const uint64_t al = ah + (L::ABYTES >> 4), bh = ah + (2 * L::ABYTES >> 4);
                    if (leader) {
                        if (i < cnt) {
                            mma_f16(d, ah, bh, mma_idesc(2 * R, 2 * L::N, true, true), i > 0);            // hi (hi | lo)
                            mma_f16(d + L::N, al, bh, mma_idesc(2 * R, L::N, true, true), 1);            // lo hi
                            mma_f16(d, ah + 16, bh + 16, mma_idesc(2 * R, 2 * L::N, true, true), 1);      // nodes 16..31
                            mma_f16(d + L::N, al + 16, bh + 16, mma_idesc(2 * R, L::N, true, true), 1);
                        }
                        mma_commit(&emptyb[i]);
                        if (i + 1 == kFoldTiles) mma_commit(&accfull[buf]);
                    }
                }
            }
        }
        // no MMA may be in flight when the tensor memory is freed
        if (leader) mma_commit(&drain[mine]);
        __syncwarp();
        if (mbar_wait(&drain[mine], 0) != WAIT_DONE) {
            timed_out = true;
            *s_abort = 1;  // (they may still read the stages, which plain_items() would reuse)
        }
    } else if (prod_index(warp) < kProd) {
        // ---------------- producers ----------------
        const int w = prod_index(warp);  // and its stage
        const unsigned half = w / kFoldTiles;
        const int slot = w % kFoldTiles;
        unsigned fb0 = 0;     // runs of this CTA's items so far
        bool stop = false;
        for (long long item = blockIdx.x; item < b.n_items && !stop; item += gridDim.x) {
            if (warp_aborted(s_abort)) break;
            const TItem it = tensor_item(b, item);
            if (!it.ok) continue;
            const int nseg = segments(it.f->n_omega, N2);
            const TensorSteps steps = it.f->steps;
            // this warp's stage is number `slot` of every second run; a short run
            // leaves it without a tile, and it is then only passed on
            const int ft = min(kFoldTiles, it.f->flush_tiles);
            const int nruns = (it.nt + ft - 1) / ft;
            auto tile_of = [&](int r) {
                const int t = r * ft + slot;
                return r < nruns && slot < ft && t < it.nt ? t : -1;
            };
            float nd[9];
            int r = (int)((fb0 ^ half) & 1), t = tile_of(r);
            if (t >= 0) load_node(*it.f, it.t0 + t, lane, nd);
            for (; r < nruns; r += 2) {
                float cur[9];
#pragma unroll
                for (int f = 0; f < 9; ++f) cur[f] = nd[f];
                const int tr = t;
                t = tile_of(r + 2);
                if (t >= 0) load_node(*it.f, it.t0 + t, lane, nd);
                // the MMAs have read the stage's last contents (the first use passes at once)
                const unsigned use = ((fb0 + r) >> 1) & 1;
                auto stage_free = [&] {
                    return warp_wait(&empty[w], use ^ 1, s_abort, b.abort, timed_out);
                };
                if (!(tr >= 0 ? produce_tile<N2, R>(smem + w * L::STAGE, cur, it, lane, nseg, steps, stage_free)
                              : stage_free())) {
                    stop = true;
                    break;
                }
                fence_proxy_async();  // this lane's operand stores, before the MMAs read them
                __syncwarp();
                if (lane == 0 && !skip_copy(b, item, tr)) mbar_arrive(&full[w]);
            }
            fb0 += nruns;
        }
    }
    if (timed_out) atomicOr(b.err, ERR_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(L::ALLOC));
    }
    // The items left over.  No role runs any more, so the words are the same for
    // every thread, and the stages are free (the MMAs' last commits have been waited for).
    if (*s_plain == 0 || *s_abort != 0) return;
    if (warp < 4) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kLaunchRegs));
    else asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kLaunchRegs));
    plain_items(b, smem, L::STAGE * kStages);
}

float2 ff(double w)
{
    const float hi = (float)w;
    return make_float2(hi, (float)(w - (double)hi));
}

template <int N2, int R>
int launch_tensor(const BatchLaunch& b, int grid, cudaStream_t s)
{
    using L = Tens<N2, R>;
    auto kern = field_tensor_kernel<N2, R>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM);
    if (e != cudaSuccess) return -(int)e;
    kern<<<grid, kTensorThreads, L::SMEM, s>>>(b);
    e = cudaGetLastError();
    return e == cudaSuccess ? 1 : -(int)e;
}

}  // namespace

// Classes: 2 omegas on each of 32 row phasors, 4 on 32, 4 on 64.
static int class_n2(int cls) { return cls == kFirstTensorClass ? 2 : 4; }

int tensor_class(int n_omega)
{
    if (n_omega < kTensorMinOmega || n_omega > kTensorMaxOmega) return -1;
    return kFirstTensorClass + (n_omega <= 64 ? 0 : (n_omega <= 128 ? 1 : 2));
}

void tensor_prepare(int cls, FieldLaunch& f)
{
    const int n2 = class_n2(cls);
    const double om0 = (double)f.om_hi0 + (double)f.om_lo0, dom = (double)f.dom_hi + (double)f.dom_lo;
    const double seed_row = 8 * seed_seg(segments(f.n_omega, n2)) + 3;
    f.steps.seed = ff(om0 + (seed_row * n2 + 0.5 * (n2 - 1)) * dom);
    f.steps.row = ff(n2 * dom);
    f.steps.seg = ff(8 * n2 * dom);
    f.steps.col = ff(0.5 * dom);
    f.steps.k0 = ff(6.283185307179586 * om0);
    f.steps.dk = ff(6.283185307179586 * dom);
}

void tensor_field_shape(int cls, int device, int* ppc, int* slots)
{
    *ppc = 1;
    switch (cls - kFirstTensorClass) {
    case 0: *slots = resident(field_tensor_kernel<2, 32>, kTensorThreads, Tens<2, 32>::SMEM, device); break;
    case 1: *slots = resident(field_tensor_kernel<4, 32>, kTensorThreads, Tens<4, 32>::SMEM, device); break;
    default: *slots = resident(field_tensor_kernel<4, 64>, kTensorThreads, Tens<4, 64>::SMEM, device);
    }
}

int launch_tensor_field(int cls, const BatchLaunch& b, int grid, cudaStream_t s)
{
    switch (cls - kFirstTensorClass) {
    case 0: return launch_tensor<2, 32>(b, grid, s);
    case 1: return launch_tensor<4, 32>(b, grid, s);
    default: return launch_tensor<4, 64>(b, grid, s);
    }
}

}  // namespace sc
