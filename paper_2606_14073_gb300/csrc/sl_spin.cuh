// sl_spin.cuh -- spin-update helpers shared by the integrator (sl_integrate.cu) and the
// self-consistent midpoint iteration (sl_midpoint.cu): the damped precession vector,
// the exact Rodrigues rotation (FP64, and an FP32 increment form), and the
// atomics-free force/field gather over an atom's own pair records.
#pragma once

#include <type_traits>

#include "sl_common.cuh"
#include "sl_eval2.cuh"
#include "sl_internal.h"

namespace sl {

template <typename R>
struct GatherArgs {
    const v4<R> *fown, *gii;
    const PairRec<R> *pd;
    const uint32_t *mask;   // in-cutoff candidate slots, [maskw][n]
    int maskw;
    int64_t n;
};

// The state arithmetic of a step names its multiply-adds: k_halves and the separate halves inline it, and a
// step's bits must not depend on which of them ran it (the compiler fuses a product and a sum as the code
// around them allows).
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
template <typename R>
__device__ __forceinline__ R cross_(R a, R b, R c, R d) { return fma_(a, b, -mul_(c, d)); }   // a b - c d
template <typename R>
__device__ __forceinline__ R dot3_(R ax, R ay, R az, R bx, R by, R bz) { return fma_(az, bz, fma_(ay, by, mul_(ax, bx))); }

template <typename R>
__device__ __forceinline__ void omega_of(R sx, R sy, R sz, R hx, R hy, R hz, R lam, R k, R w[3]) {
    w[0] = mul_(fma_(lam, cross_(sy, hz, sz, hy), hx), k);
    w[1] = mul_(fma_(lam, cross_(sz, hx, sx, hz), hy), k);
    w[2] = mul_(fma_(lam, cross_(sx, hy, sy, hx), hz), k);
}

__device__ __forceinline__ void rotate(double sx, double sy, double sz, const double w[3], double dt, double out[3]) {
    const double wn2 = dot3_(w[0], w[1], w[2], w[0], w[1], w[2]);
    if (wn2 == 0.0) { out[0] = sx; out[1] = sy; out[2] = sz; return; }
    const double wn = sqrt(wn2);
    const double ax = w[0] / wn, ay = w[1] / wn, az = w[2] / wn;
    double s, c;
    sincos(mul_(wn, dt), &s, &c);
    const double p = mul_(dot3_(ax, ay, az, sx, sy, sz), 1.0 - c);
    out[0] = fma_(ax, p, fma_(cross_(ay, sz, az, sy), s, mul_(sx, c)));
    out[1] = fma_(ay, p, fma_(cross_(az, sx, ax, sz), s, mul_(sy, c)));
    out[2] = fma_(az, p, fma_(cross_(ax, sy, ay, sx), s, mul_(sz, c)));
}

// Rotation increment dS = Rot(S, w dt) - S in FP32 (added to the FP64 spin by the
// caller): dS = (a x S) sin(th) - 2 sin^2(th/2) (S - a (a.S)), th = |w| dt.
__device__ __forceinline__ void rotate_delta_f(float sx, float sy, float sz, float wx, float wy, float wz, float dt,
                                               float d[3]) {
    const float wn2 = dot3_(wx, wy, wz, wx, wy, wz);
    if (wn2 == 0.0f) { d[0] = d[1] = d[2] = 0.0f; return; }
    const float iw = rsqrtf(wn2);
    const float ax = mul_(wx, iw), ay = mul_(wy, iw), az = mul_(wz, iw);
    float sh, ch;
    sincosf(mul_(mul_(mul_(0.5f, wn2), iw), dt), &sh, &ch);
    const float sn = mul_(2.0f * sh, ch), omc = mul_(2.0f * sh, sh);
    const float as = dot3_(ax, ay, az, sx, sy, sz);
    d[0] = cross_(cross_(ay, sz, az, sy), sn, omc, fma_(-ax, as, sx));
    d[1] = cross_(cross_(az, sx, ax, sz), sn, omc, fma_(-ay, as, sy));
    d[2] = cross_(cross_(ax, sy, ay, sx), sn, omc, fma_(-az, as, sz));
}

// F_k = sum_j dE_k/dr_kj - sum_j dE_j/dr_jk, H_k = -dE_k/dS_k - sum_j dE_j/dS_k: the
// records (dE_j/dr_jk, dE_j/dS_k) sit in k's own in-cutoff candidate slots.  W lanes take an atom;
// lane q walks the slots s = q mod W in order with the other lanes of its warp, so the records
// that neighbouring atoms read at one slot are neighbours in memory (slot-major layout); the
// lanes' sums are added in a fixed order.  What bounds it: the records' DRAM traffic in large FP32 systems
// (2.3 GB in 470 us at 884,736 atoms), and elsewhere the chain of a lane's slots, a few loads in flight
// at a time: so several slots' records are loaded together, without branches, eight with one or four lanes per
// atom and four with eight, which have no more of a mask word (FP64 at 32,768 atoms 92 instead of 120 us a
// second half, FP32 at 110,592 83 instead of 85), and a
// small system (gather_lanes) takes several lanes per atom, a larger one one.  Second half, mixed
// precision, 512 / 13,824 / 32,768 / 64,000 / 110,592 atoms: 15 / 19 / 37 us at the first three with eight lanes, 17 /
// 21 / 32 / 59 / 89 with four, 27 / 31 / 43 / 59 / 83 with one; FP64, 512 / 13,824 / 21,952 / 32,768 atoms: 27 / 49 / 77 / 114 us with
// eight, 83 / 87 / 88 / 92 with one.  The eight lanes' line is one for both precisions, near where mixed
// precision's four lanes catch up; FP64's own crossing lies between 21,952 and 32,768 atoms.
constexpr int gather_atoms(int W) { return 256 / W; }   // atoms per 256-thread block
inline int gather_lanes(const Sys &s) { return s.n <= 16384 ? 8 : s.prec != 0 && s.n <= 65536 ? 4 : 1; }
// launch(W) with the system's W (R: its precision) as a constant
template <typename R, typename F>
inline void with_gather_lanes(const Sys &s, F launch) {
    const int w = gather_lanes(s);
    if (w == 8) launch(std::integral_constant<int, 8>());
    else if (w == 1) launch(std::integral_constant<int, 1>());
    else if constexpr (sizeof(R) == 4) launch(std::integral_constant<int, 4>());
}

template <typename R, int W>
struct GatherSmem {
    R v[W == 1 ? 1 : 6][W == 1 ? 1 : gather_atoms(W)];   // (unused with one lane per atom)
};

// The record at p where it is set, else zeros, without a branch, so the loads of several slots are in
// flight together: FP32 in one 256-bit load, FP64 in two.
__device__ __forceinline__ PairRec<float> rec_if(const PairRec<float> *p, uint32_t set) {
    PairRec<float> e = {};
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %9, 0;\n\t@p ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t}"
        : "+f"(e.a.x), "+f"(e.a.y), "+f"(e.a.z), "+f"(e.a.w), "+f"(e.b.x), "+f"(e.b.y), "+f"(e.b.z), "+f"(e.b.w)
        : "l"(p), "r"(set));
    return e;
}
__device__ __forceinline__ PairRec<double> rec_if(const PairRec<double> *p, uint32_t set) {
    PairRec<double> e = {};
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %7, 0;\n\t@p ld.global.v4.f64 {%0, %1, %2, %3}, [%6];\n\t"
        "@p ld.global.v2.f64 {%4, %5}, [%6 + 32];\n\t}"
        : "+d"(e.a.x), "+d"(e.a.y), "+d"(e.a.z), "+d"(e.a.w), "+d"(e.b.x), "+d"(e.b.y)
        : "l"(p), "r"(set));
    return e;
}

// Sums of one atom's own part and records, its lane q of W.
template <typename R, int W>
__device__ __forceinline__ void gather_lane(const GatherArgs<R> &g, int64_t k, int q, R v[6]) {
    const int64_t N = g.n;
#pragma unroll
    for (int c = 0; c < 6; ++c) v[c] = R(0);
    if (q == 0) {
        const v4<R> fo = ro(g.fown + k), gi = ro(g.gii + k);
        v[0] = fo.x; v[1] = fo.y; v[2] = fo.z;
        v[3] = -gi.x; v[4] = -gi.y; v[5] = -gi.z;
    }
#pragma unroll 1
    for (int w = 0; w < g.maskw; ++w) {
        const uint32_t word = ro(g.mask + (int64_t)w * N + k);
        constexpr int U = 4 * W <= 16 ? 8 : 4;   // slots at a time
#pragma unroll 1
        for (int b = q; b < 32; b += U * W) {
            if ((word >> b) == 0u) break;
            PairRec<R> e[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                e[u] = rec_if(g.pd + (int64_t)(w * 32 + b + u * W) * N + k, (word >> (b + u * W)) & 1u);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                v[0] -= e[u].a.x; v[1] -= e[u].a.y; v[2] -= e[u].a.z;
                v[3] -= e[u].a.w; v[4] -= e[u].b.x; v[5] -= e[u].b.y;
            }
        }
    }
}

// The atoms of block blk (blockDim.x / W of them): the atom of this thread (-1: none) and its sums F, H.
template <typename R, int W>
__device__ __forceinline__ int64_t gather_block(const GatherArgs<R> &g, int64_t blk, GatherSmem<R, W> &sm, double F[3],
                                                double H[3]) {
    const int per = blockDim.x / W;
    const int64_t i = blk * per + threadIdx.x;   // the thread's atom afterwards
    R v[6];
    if constexpr (W == 1) {
        if (i >= g.n) return -1;
        gather_lane<R, 1>(g, i, 0, v);
    } else {
        const int at = threadIdx.x / W, q = threadIdx.x % W;
        const int64_t k = blk * per + at;
        gather_lane<R, W>(g, k < g.n ? k : g.n - 1, q, v);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
#pragma unroll
            for (int o = 1; o < W; o <<= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
            if (q == 0) sm.v[c][at] = v[c];
        }
        __syncthreads();
        if (threadIdx.x >= per || i >= g.n) return -1;
#pragma unroll
        for (int c = 0; c < 6; ++c) v[c] = sm.v[c][threadIdx.x];
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        F[c] = (double)v[c];
        H[c] = (double)v[3 + c];
    }
    return i;
}

}  // namespace sl
