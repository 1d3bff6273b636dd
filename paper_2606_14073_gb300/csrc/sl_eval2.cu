// sl_eval2.cu -- NEP-SPIN evaluation: compacted radial kernels and quad-per-atom angular kernels.
//
// Same mathematics as the descriptor of arXiv 2606.14073 (Sections 5.1.1-5.1.2, 5.2.3-5.2.4)
// described in sl_nep.cu; this file maps it onto the GPU differently:
//
//   k_crad     one thread per atom, one pass over the candidate list (which carries a
//              skin): compacts the pairs inside the cutoffs into angular rows
//              (r < rc_ang) and radial-only rows (rc_ang <= r < rc_rad), each grouped by
//              neighbour species, and accumulates the radial and pairwise-magnetic basis
//              sums over them, contracted with the coefficients once per neighbour
//              species (q^R, q^EX, q^DMI, q^ANI, q^SIA, q^O).
//   k_crad_wide  the same with sixteen lanes per atom (small systems, and FP64); in the smallest ones as
//              k_crad_rows (compaction) and k_crad_sums, beside the angular kernel.
//   k_ang_fwd  four lanes per atom (k_ang_wide: a warp, in small systems).  Each lane stages one angular pair
//              (carrier, g_n, spin weight, the 24 solid harmonics) in shared memory; then
//              every lane accumulates B_nlm, BS_nlm for its 6 harmonics over the staged pairs.
//   k_bwd      four lanes per atom (k_bwd_wide: a warp), lanes over pairs.  The angular adjoints
//              dE/dB_nlm = 2 kappa_lm Fp B_nlm and the precontracted radial
//              coefficients of the atom sit in shared memory; each lane takes whole
//              pairs (angular rows first, then radial-only rows) and writes the pair
//              record (dE_i/dr_ij, dE_i/dS_j) straight into the slot the neighbour j
//              will read (its own list slot of i); the per-atom sums (dE_i/dr_i side,
//              dE_i/dS_i, virial) are reduced over the quad.
// The force/field gather (sl_integrate.cu) then reads, for atom k, the records of
// its in-cutoff slots only.
#include <cstddef>
#include <mutex>
#include <vector>

#include "sl_internal.h"
#include "sl_eval2.cuh"
#include "sl_batch.h"
#include "sl_fused.cuh"

namespace sl {

// ------------------------------------------------------------------ helpers
// Two independent multiply-adds per instruction where the hardware has them (FP32 pairs:
// the packed FMA of sm_100 and later; each component rounds like fmaf), plain FMAs in FP64.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
template <typename R>
__device__ __forceinline__ v2<R> pair2(R x, R y) {
    v2<R> v;
    v.x = x;
    v.y = y;
    return v;
}
// FP32: the carrier f_k = (T_k(x) + 1) f_c/2 as pairs of neighbouring k, k = 8 last: T_{k+2} = 2 T_2 T_k -
// T_{k-2} advances two k's per packed multiply-add, and sums over pairs by k need no f_k twice in a
// register pair.  (T_4 .. T_7 are carried negated, which saves the recurrence its sign changes.)
struct CarrierPairs {
    float2 f[4];
    float f8;
    __device__ __forceinline__ CarrierPairs(float r, float inv_rc) {
        const float t = r * inv_rc, fch = cut_half(t);
        const float y = t - 1.f, x = fma_(2.f * y, y, -1.f), x2 = 2.f * x;
        const float t2 = fma_(x2, x, -1.f), w = 2.f * t2;
        const float2 s0 = make_float2(1.f, x), s1 = make_float2(t2, fma_(x2, t2, -x));
        const float2 s2 = fma2(make_float2(-w, -w), s1, s0), s3 = fma2(make_float2(w, w), s2, s1);
        const float2 F = make_float2(fch, fch), Fm = make_float2(-fch, -fch);
        f[0] = make_float2(fch + fch, fma_(x, fch, fch));
        f[1] = fma2(s1, F, F);
        f[2] = fma2(s2, Fm, F);
        f[3] = fma2(s3, Fm, F);
        f8 = fma_(fma_(-w, s3.x, s2.x), fch, fch);
    }
};

template <typename R>
__device__ __forceinline__ v4<R> quad4(const v2<R> &a, const v2<R> &b) {
    v4<R> v;
    v.x = a.x; v.y = a.y; v.z = b.x; v.w = b.y;
    return v;
}
// The carrier of sl_common.cuh with the T_k and U_k recurrences advanced together (FP32).
template <typename R>
__device__ __forceinline__ void carrier_fd2(R r, R inv_rc, R f[NK], R df[NK]) {
    const R t = r * inv_rc;
    R fch, dfch;
    cut_half_d(t, inv_rc, fch, dfch);
    const R y = t - R(1);
    const R x = R(2) * y * y - R(1);
    const R dxr = R(4) * y * inv_rc;
    const R x2 = R(2) * x;
    const R dxf = dxr * fch;
    v2<R> tum = pair2<R>(R(1), R(1)), tuc = pair2<R>(x, x2);   // (T_0, U_0), (T_1, U_1)
    f[0] = R(2) * fch;
    df[0] = R(2) * dfch;
    f[1] = fma_(x, fch, fch);
    df[1] = dxf + fma_(x, dfch, dfch);
#pragma unroll
    for (int k = 2; k < NK; ++k) {
        const v2<R> tun = fma2(pair2<R>(x2, x2), tuc, pair2<R>(-tum.x, -tum.y));
        f[k] = fma_(tun.x, fch, fch);
        df[k] = fma_(R(k) * tuc.y, dxf, fma_(tun.x, dfch, dfch));
        tum = tuc;
        tuc = tun;
    }
}

// g_n = sum_k c_nk f_k and dg_n = sum_k c_nk df_k together, two multiply-adds per instruction
template <typename R, int TI, int TJ, int G>
__device__ __forceinline__ void contract_k2(const NepDev<R> &P, const R f[NK], const R df[NK], R g[NCH], R dg[NCH]) {
#pragma unroll
    for (int n = 0; n < NCH; ++n) {
        v2<R> s = pair2<R>(R(0), R(0));
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            const R c = P.c[TI][TJ][G][n][k];
            s = fma2(pair2<R>(c, c), pair2<R>(f[k], df[k]), s);
        }
        g[n] = s.x;
        dg[n] = s.y;
    }
}

// FP64: the radial carrier f_k = (T_k(x) + 1) f_c/2 at r: x and 2x, f_c/2 and its slope, dx/dr f_c/2.
// A contraction sum_k C_k f_k is f_c/2 times P = sum_k C_k (T_k + 1), and its slope
// d(f_c/2)/dr P + dx/dr f_c/2 Q with Q = sum_k C_k dT_k/dx, dT_k/dx = k U_{k-1}; with C_0 replaced
// by 2 C_0 + sum_{k>0} C_k (shifted coefficients) P is sum_k C_k T_k.  So no f_k or df_k is
// formed: 28 of 270 FP64 instructions of a radial pair less.  (FP32 keeps f_k and df_k: with its
// registers capped at 128 this form, whose partial sums live longer, ran the backward at 1.60
// instead of 1.58 ms at 884,736 atoms.)
template <typename R>
struct Carrier {
    R x, x2, fch, dfch, dxf;
    __device__ __forceinline__ Carrier(R r, R inv_rc) {
        const R t = r * inv_rc;
        cut_half_d(t, inv_rc, fch, dfch);
        const R y = t - R(1);
        x = R(2) * y * y - R(1);
        x2 = R(2) * x;
        dxf = R(4) * y * inv_rc * fch;
    }
    // use(k, (T_k, dT_k/dx)) for k = 2 .. NK - 1
    template <typename F>
    __device__ __forceinline__ void terms(F use) const {
        v2<R> m = pair2<R>(R(1), R(1)), c = pair2<R>(x, x2);   // (T_{k-2}, U_{k-2}), (T_{k-1}, U_{k-1})
#pragma unroll
        for (int k = 2; k < NK; ++k) {
            const v2<R> n = fma2(pair2<R>(x2, x2), c, pair2<R>(-m.x, -m.y));
            use(k, pair2<R>(n.x, R(k) * c.y));
            m = c;
            c = n;
        }
    }
};

template <typename R, int TI, int TJ, int G>
__device__ __forceinline__ void contract_k(const NepDev<R> &P, const R f[NK], R g[NCH]) {
#pragma unroll
    for (int n = 0; n < NCH; ++n) {
        R s = R(0);
#pragma unroll
        for (int k = 0; k < NK; ++k) s += P.c[TI][TJ][G][n][k] * f[k];
        g[n] = s;
    }
}

// Atom j's position and spin: FP32 interleaved, one 256-bit load (a neighbour's 32-byte sector holds both:
// the backward at 884,736 atoms 1.40 instead of 1.49 ms, the angular kernel 474 instead of 483 us); FP64
// two arrays.  The cutoff tests, which need no spin, read the positions alone (the radial kernel's
// from the interleaved array: 993 instead of 882 us).
__device__ __forceinline__ void pair_at(const Eval2Args<float> &a, int64_t j, float4 &p, float4 &s) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(p.x), "=f"(p.y), "=f"(p.z), "=f"(p.w), "=f"(s.x), "=f"(s.y), "=f"(s.z), "=f"(s.w)
        : "l"(a.pos + 2 * j));
}
__device__ __forceinline__ void pair_at(const Eval2Args<double> &a, int64_t j, double4 &p, double4 &s) {
    p = ro(a.pos + j);
    s = ro(a.spin + j);
}

template <typename R>
__device__ __forceinline__ void sep(const BoxDev<R> &b, const v4<R> &pi, const v4<R> &pj, R &dx, R &dy, R &dz) {
    dx = pj.x - pi.x;
    dy = pj.y - pi.y;
    dz = pj.z - pi.z;
    minimg(b, dx, dy, dz);
}

// Coefficients of the rc_rad groups (g in the order R, EX, DMI, ANI, SIA) for lanes that each take
// their own: for the wide radial kernel's contraction [centre][neighbour][k][g * 5 + n], rows
// padded to 32, then for the backward's precontraction [centre][neighbour][n][group][k], rows of 12, the
// groups in the order EX, DMI, ANI, SIA, R (FP64: k = 0 shifted, see Carrier).
constexpr int CTAB_BWD = NS * NS * NK * 32, CB_ROW = 12, CB_CENTRE = NS * NCH * 5 * CB_ROW;
template <typename R>
static void fill_ctab(const NepDev<R> &P, std::vector<R> &t) {
    constexpr int GG[5] = {G_R, G_EX, G_DMI, G_ANI, G_SIA};
    t.assign((size_t)CTAB_BWD + NS * CB_CENTRE, R(0));
    for (int x = 0; x < NS; ++x)
        for (int y = 0; y < NS; ++y)
            for (int o = 0; o < 25; ++o) {
                const R *c = P.c[x][y][GG[o / NCH]][o % NCH];
                R *b = t.data() + CTAB_BWD + (size_t)(((x * NS + y) * NCH + o % NCH) * 5 + (o / NCH + 4) % 5) * CB_ROW;
                for (int k = 0; k < NK; ++k) t[(size_t)((x * NS + y) * NK + k) * 32 + o] = b[k] = c[k];
                if (sizeof(R) == 8) b[0] = R(shifted_c0(c));
            }
}
int make_coeff_table(Sys &s) {
    const auto put = [&](const auto &t) {
        const size_t bytes = t.size() * sizeof(t[0]);
        if (!s.ctab && cudaMalloc(&s.ctab, bytes) != cudaSuccess) {
            s.ctab = nullptr;
            return -1;
        }
        if (cudaMemcpyAsync(s.ctab, t.data(), bytes, cudaMemcpyHostToDevice, s.stream) != cudaSuccess) return -1;
        return cudaStreamSynchronize(s.stream) == cudaSuccess ? 0 : -1;
    };
    if (s.prec == 0) {
        std::vector<double> t;
        fill_ctab(s.pd, t);
        return put(t);
    }
    std::vector<float> t;
    fill_ctab(s.pf, t);
    return put(t);
}

// harmonic m of lane ql of an atom's LPA: four lanes take neighbouring pairs (2 ql, 2 ql + 1, then eight
// further, so that a pair of records is whole 16-byte pieces), a warp one each
template <int LPA>
__device__ __forceinline__ constexpr int lm_of(int ql, int m) {
    static_assert(LPA == 4 || LPA == 32, "24 harmonics in equal shares, or one per lane");
    return LPA == 4 ? 2 * ql + (m & 1) + 8 * (m >> 1) : ql;
}
__device__ __forceinline__ int l_of_lm(int lm) { return lm < 3 ? 1 : lm < 8 ? 2 : lm < 15 ? 3 : 4; }
template <typename R>
__device__ __forceinline__ R kappa_of_lm(int lm) {
    // kappa_lm of the addition theorem, selected at run time (the quad lane picks its harmonics)
    switch (lm) {
    case 0: case 1: case 2: return R(1.0);
    case 3: case 4: case 5: return R(3.0);
    case 6: return R(0.75);
    case 7: return R(0.25);
    case 8: return R(0.625);
    case 9: return R(15.0);
    case 10: return R(0.375);
    case 11: return R(0.25);
    case 12: return R(0.375);
    case 13: return R(3.75);
    case 14: return R(0.625);
    case 15: return R(8.75);
    case 16: return R(4.375);
    case 17: return R(1.25);
    case 18: return R(0.625);
    case 19: return R(0.015625);
    case 20: return R(0.625);
    case 21: return R(0.3125);
    case 22: return R(4.375);
    default: return R(0.546875);
    }
}

// ------------------------------------------------------------------ k_crad
// One thread per atom (mixed precision, larger systems: see crad_is_wide), per neighbour species:
//  A. the angular candidates (within rc_ang + skin of the list build, so nearly all inside
//     rc_rad): compaction and the radial and pairwise-magnetic basis sums in one pass;
//  B. the radial-shell candidates (rc_ang + skin .. rc_rad + skin at the build, fewer than
//     half inside rc_rad): compaction only, a few instructions per candidate;
//  C. the basis sums over the rows B produced.
// Splitting B from C keeps a warp from running the pair arithmetic for every candidate of
// the shell whenever one of its 32 atoms has that candidate inside the cutoff.  Rows are
// angular (r < rc_ang) or radial-only (rc_ang <= r < rc_rad), each in candidate order (the
// candidates of neighbour species 0 come first in a list, then those of species 1), for the
// angular and backward kernels and the gather.  The sums are
// contracted with the coefficients once per neighbour species (q^R, q^EX, q^DMI, q^ANI,
// q^SIA); q^O = |S|^2.
// What bounds it: latency, at 16 warps per SM (the sums take 45 of 128 registers): 50% of issue slots, no
// unit above 56% (0.78 ms at 884,736 atoms on a crystal, 1.00 ms after 600 steps at 300 K, when a warp's atoms
// have uneven lists).  So the loads are kept in flight: the next candidate's coordinates in A, the next
// four's in B, the next row's in C, and the first species' 25 values all at once before the second's
// are stored (each load behind the store before it cost 25 trips to the L2 cache): 921 to 881 us at
// 884,736 atoms, 161 to 147 us at 110,592 (two candidates ahead in A: 898 and 147 us; A as four at a
// time, loaded where they are used: 926 and 150 us).  Lists tiled so that a warp's list loads are
// consecutive changed nothing (936 us).

struct RadSums {
    float2 b[5][4];   // R, EX, DMI, ANI, SIA sums of k = 0 .. 7, two per packed multiply-add
    float b8[5];      // k = 8
    __device__ __forceinline__ float at(int g, int k) const { return k == 8 ? b8[g] : k & 1 ? b[g][k / 2].y : b[g][k / 2].x; }
};

__device__ __forceinline__ void rad_accumulate(const NepDev<float> &P, const float4 &si, const float4 &cs, float dx,
                                               float dy, float dz, float d2, RadSums &b) {
    const float ir = rsqrt_(d2), r = d2 * ir;
    const float ux = dx * ir, uy = dy * ir, uz = dz * ir;
    const CarrierPairs cr(r, P.inv_rc_r);
    const float sij = si.x * cs.x + si.y * cs.y + si.z * cs.z;
    const float siu = si.x * ux + si.y * uy + si.z * uz;
    const float sju = cs.x * ux + cs.y * uy + cs.z * uz;
    const float dmi = (si.y * cs.z - si.z * cs.y) * ux + (si.z * cs.x - si.x * cs.z) * uy + (si.x * cs.y - si.y * cs.x) * uz;
    const float h[5] = {1.f, sij, dmi, siu * sju, siu * siu};
#pragma unroll
    for (int g = 0; g < 5; ++g) {
#pragma unroll
        for (int p = 0; p < 4; ++p)
            b.b[g][p] = g == 0 ? __fadd2_rn(cr.f[p], b.b[g][p]) : fma2(cr.f[p], make_float2(h[g], h[g]), b.b[g][p]);
        b.b8[g] = g == 0 ? b.b8[g] + cr.f8 : fma_(cr.f8, h[g], b.b8[g]);
    }
}

// Row of an in-cutoff pair, or -1 (angular rows full: only after a list overflow, which ovf
// records; the atom reports it once its rows are written).
template <typename R>
__device__ __forceinline__ int take_row(const NepDev<R> &P, const Eval2Args<R> &a, R d2, int &na, int &nr,
                                        bool &ovf) {
    if (d2 < P.rc_a2) {
        if (na >= a.cap_ang) {
            ovf = true;
            return -1;
        }
        return na++;
    }
    return a.cap_ang + nr++;
}

// in-cutoff slot bits of this thread's atom, in shared memory (column threadIdx.x)
constexpr int MASKW_MAX = 8;   // slot-mask words (a list holds at most 256 candidates)
__device__ __forceinline__ void mark_slot(uint32_t (*sm)[128], int slot) {
    sm[slot >> 5][threadIdx.x] |= 1u << (slot & 31);
}

template <typename R, int TI, int TJ>
__device__ __forceinline__ void crad_species(const NepDev<R> &P, const Eval2Args<R> &a, int64_t i, const v4<R> &pi,
                                             const v4<R> &si, int lo0, int hi0, int lo1, int hi1, int &na, int &nr,
                                             bool &ovf, uint32_t (*smask)[128]) {
    RadSums b;
#pragma unroll
    for (int g = 0; g < 5; ++g) {
        b.b8[g] = 0.f;
#pragma unroll
        for (int p = 0; p < 4; ++p) b.b[g][p] = make_float2(0.f, 0.f);
    }
    const int64_t N = a.n;
    // this atom's candidate list and reverse slots: one row each, read in aligned chunks of 4
    // entries (a 16-byte and a 4-byte load), two chunks ahead of the one being tested
    const int32_t *__restrict__ nrow = a.nbr + i * a.capr;
    const uint8_t *__restrict__ rrow = a.rev + i * a.capr;
    auto chunk = [&](int c, int hi, int4 &jq, uchar4 &tq) {
        if (c < hi) {
            jq = *reinterpret_cast<const int4 *>(nrow + c);
            tq = *reinterpret_cast<const uchar4 *>(rrow + c);
        }
    };

    // A: angular candidates, compaction and sums; the coordinates of the next candidate are in flight
    // while one is computed
    {
        int4 jq1 = make_int4(-1, -1, -1, -1), jq2 = jq1;
        uchar4 tq1 = make_uchar4(0, 0, 0, 0), tq2 = tq1;
        const int c0 = lo0 & ~3;
        chunk(c0, hi0, jq1, tq1);
        chunk(c0 + 4, hi0, jq2, tq2);
        auto pick = [&](int c, int j) { return c >= lo0 && c < hi0 ? j : (int)i; };   // not another segment's entry
        const int ja = pick(c0, jq1.x);
        v4<R> p1, s1;
        pair_at(a, ja, p1, s1);
#pragma unroll 1
        for (int c = c0; c < hi0; c += 4) {
            const int jj[5] = {jq1.x, jq1.y, jq1.z, jq1.w, jq2.x};
            const int tt[4] = {tq1.x, tq1.y, tq1.z, tq1.w};
            jq1 = jq2;
            tq1 = tq2;
            chunk(c + 8, hi0, jq2, tq2);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const v4<R> pu = p1, su = s1;
                const int jn = pick(c + u + 1, jj[u + 1]);
                pair_at(a, jn, p1, s1);
                if (c + u < lo0 || c + u >= hi0) continue;
                R dx, dy, dz;
                sep(a.box, pi, pu, dx, dy, dz);
                const R d2 = dx * dx + dy * dy + dz * dz;
                if (!(d2 < P.rc_r2)) continue;
                const int row = take_row(P, a, d2, na, nr, ovf);
                if (row < 0) continue;
                stg(a.crow + (int64_t)row * N + i, make_int2(jj[u], tt[u]));
                mark_slot(smask, c + u);
                rad_accumulate(P, si, su, dx, dy, dz, d2, b);
            }
        }
    }
    // B: radial-shell candidates, compaction only; the next four candidates' positions are in flight
    const int naB = na, nrB = nr;
    {
        int4 jq1 = make_int4(-1, -1, -1, -1), jq2 = jq1;
        uchar4 tq1 = make_uchar4(0, 0, 0, 0), tq2 = tq1;
        const int c0 = lo1 & ~3;
        chunk(c0, hi1, jq1, tq1);
        chunk(c0 + 4, hi1, jq2, tq2);
        auto pick = [&](int c, int j) { return c >= lo1 && c < hi1 ? j : (int)i; };
        v4<R> pn[4];
        {
            const int j[4] = {jq1.x, jq1.y, jq1.z, jq1.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) pn[u] = a.posf[pick(c0 + u, j[u])];
        }
#pragma unroll 1
        for (int c = c0; c < hi1; c += 4) {
            const int jj[4] = {jq1.x, jq1.y, jq1.z, jq1.w}, jx[4] = {jq2.x, jq2.y, jq2.z, jq2.w};
            const int tt[4] = {tq1.x, tq1.y, tq1.z, tq1.w};
            jq1 = jq2;
            tq1 = tq2;
            chunk(c + 8, hi1, jq2, tq2);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const v4<R> pu = pn[u];
                pn[u] = a.posf[pick(c + 4 + u, jx[u])];
                if (c + u < lo1 || c + u >= hi1) continue;
                R dx, dy, dz;
                sep(a.box, pi, pu, dx, dy, dz);
                const R d2 = dx * dx + dy * dy + dz * dz;
                if (!(d2 < P.rc_r2)) continue;
                const int row = take_row(P, a, d2, na, nr, ovf);
                if (row < 0) continue;
                stg(a.crow + (int64_t)row * N + i, make_int2(jj[u], tt[u]));
                mark_slot(smask, c + u);
            }
        }
    }
    // C: sums over the rows B wrote (angular rows naB..na, rare, then radial-only rows),
    // with the list entry two rows ahead and the coordinates of the next row in flight
    {
        const int nA = na - naB, len = nA + (nr - nrB);
        auto row_of = [&](int t) { return t < nA ? naB + t : a.cap_ang + nrB + (t - nA); };
        int j1 = 0, j2 = 0;
        v4<R> p1, s1;
        if (len > 0) j1 = a.crow[(int64_t)row_of(0) * N + i].x;
        if (len > 1) j2 = a.crow[(int64_t)row_of(1) * N + i].x;
        if (len > 0) pair_at(a, j1, p1, s1);
#pragma unroll 1
        for (int t = 0; t < len; ++t) {
            const v4<R> pj = p1, sj = s1;
            if (t + 1 < len) pair_at(a, j2, p1, s1);
            if (t + 2 < len) j2 = a.crow[(int64_t)row_of(t + 2) * N + i].x;
            R dx, dy, dz;
            sep(a.box, pi, pj, dx, dy, dz);
            rad_accumulate(P, si, sj, dx, dy, dz, dx * dx + dy * dy + dz * dz, b);
        }
    }
    // contraction of this species' sums; the second species adds onto the first's
    // values in q (the same thread wrote them), so no accumulator lives across the loops
    constexpr int GQ[5] = {Q_R, Q_EX, Q_DMI, Q_ANI, Q_SIA};
    constexpr int GG[5] = {G_R, G_EX, G_DMI, G_ANI, G_SIA};
    R first[5][NCH];   // all loads before the first store: the stores keep their order
#pragma unroll
    for (int g = 0; g < 5; ++g)
#pragma unroll
        for (int n = 0; n < NCH; ++n) first[g][n] = TJ == 0 ? R(0) : a.q[(GQ[g] + n) * a.qs + i];
#pragma unroll
    for (int g = 0; g < 5; ++g) {
#pragma unroll
        for (int n = 0; n < NCH; ++n) {
            R v = first[g][n];
#pragma unroll
            for (int k = 0; k < NK; ++k) v += P.c[TI][TJ][GG[g]][n][k] * b.at(g, k);
            stg(a.q + (GQ[g] + n) * a.qs + i, v);
        }
    }
}

template <typename R, int TI>
__device__ __forceinline__ void crad_atom(const NepDev<R> &P, const Eval2Args<R> &a, int64_t i,
                                          uint32_t (*smask)[128]) {
    const int64_t N = a.n;
    v4<R> pi, si;
    pair_at(a, i, pi, si);
    const int4 sg = a.seg[i];
    int na = 0, nr = 0;
    bool ovf = false;
    for (int w = 0; w < a.maskw; ++w) smask[w][threadIdx.x] = 0u;
    crad_species<R, TI, 0>(P, a, i, pi, si, 0, sg.x, sg.x, sg.y, na, nr, ovf, smask);
    const int na0 = na, nr0 = nr;
    crad_species<R, TI, 1>(P, a, i, pi, si, sg.y, sg.z, sg.z, sg.w, na, nr, ovf, smask);
    if (ovf) atomicOr(a.status, ST_NBR_OVERFLOW);
    stg(a.cnt + i, make_int4(na0, na, nr0, nr));
    for (int w = 0; w < a.maskw; ++w) stg(reinterpret_cast<int *>(a.mask) + (int64_t)w * N + i, (int)smask[w][threadIdx.x]);
    stg(a.q + Q_O * a.qs + i, si.x * si.x + si.y * si.y + si.z * si.z);
}

// MINB: minimum resident blocks per SM the register allocation is held to (the autotuner's
// register-budget dimension); the default is the first value of each kernel's list below.
template <typename R>
__device__ __forceinline__ void crad_body(const NepDev<R> &P, const Eval2Args<R> &args, int64_t blk,
                                          uint32_t (*smask)[128]) {
    // the arguments as values: read once from the block's copy, so nothing in the loops below
    // depends on where they are stored
    const Eval2Args<R> a = args;
    if (a.skip && *a.skip) return;
    const int64_t i = blk * (int64_t)blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    if (i < a.n_fe) crad_atom<R, 0>(P, a, i, smask);
    else crad_atom<R, 1>(P, a, i, smask);
}

// ------------------------------------------------------------------ k_crad_wide
// Sixteen lanes per atom, two atoms per warp: every FP64 system, and mixed-precision systems of
// up to CRAD_WIDE_MAX atoms.
//  A. sixteen candidates at a time, in list order: cutoff test, rows written (ballot/popc), the
//     neighbour kept in the atom's shared list (grouped by species, as the candidates are);
//  B. sixteen pairs of that list at a time: each lane takes one pair (geometry, carrier, spin
//     products) and stages it; then lane (two k's, third) adds every third staged pair into its
//     ten basis sums (five groups, two k's), one set per neighbour species;
//  C. the thirds are added, and the lanes contract the 2 x 45 sums with the coefficients.
// Rows are angular (r < rc_ang) or radial-only, in the angular and backward kernels' order.
// What bounds it.  FP64: the FP64 pipe (360 warp instructions per atom, as many as one thread per
// atom takes, but spread over a warp for every two atoms): 512 / 13,824 / 110,592 atoms 45 / 349 /
// 2,113 us, against 511 / 525 / 2,091 us with one thread per atom.  Mixed precision: instruction
// issue (1,270 warp instructions per atom against 570 for one thread per atom, whose chain of 110
// candidates takes 47 us however few the atoms): 512 / 13,824 / 32,768 / 110,592 atoms 15 / 35 / 70 /
// 202 us, against 47 / 64 / 72 / 148 us.  The line lies at 16,384 atoms, below the crossing: a
// replica keeps its kernel in a batch (its results are the same there bit for bit), where other
// replicas fill the GPU and only the instructions count (eight replicas of 4,096 to 65,536 atoms
// step 2.5% slower with the line at 32,768).
constexpr int CR_LANES = 16;             // lanes per atom
constexpr int CR_LD = 20;                // staged pair: f_0..f_8, three pads, sij, dmi, ani, sia, pads
constexpr int CR_STAGE = CR_LANES * CR_LD + 16;   // the pad puts a warp's two atoms in different banks
constexpr int CR_NQ = 26;                // descriptor entries an atom gets here

// Test of the candidate pair (i, j), j's FP32 position at hand: inside rc_rad, inside rc_ang.  FP32: on the FP32
// positions.  FP64: an FP32 separation decides outside the rounding band around a cutoff and
// the FP64 test inside it; the FP64 pipe (two lanes per SM and cycle) would otherwise spend a
// seventh of the kernel on the test.
template <typename R>
struct CradTest;
template <>
struct CradTest<float> {
    float4 pi;
    __device__ __forceinline__ CradTest(const NepDev<float> &, const Eval2Args<float> &a, int64_t i) : pi(a.posf[i]) {}
    __device__ __forceinline__ void operator()(const NepDev<float> &P, const Eval2Args<float> &a, int, const float4 &fj,
                                               bool &in, bool &ang) const {
        float dx, dy, dz;
        sep(a.box, pi, fj, dx, dy, dz);
        const float d2 = dx * dx + dy * dy + dz * dz;
        in = d2 < P.rc_r2;
        ang = d2 < P.rc_a2;
    }
};
template <>
struct CradTest<double> {
    double4 pi;
    float4 fi;
    float band;
    // Band: the FP32 copies are off by 2^-24 of themselves and the separation's own rounding and
    // minimum image add as much of the coordinates and of a box length, so a component of a
    // near pair's separation is off by at most E = 2^-24 (8 |x_i| + 4 L + 64) (the pair's other
    // coordinate is within a box length and a few A of x_i), and d2 by 2 sqrt(3) R E + 3 E^2 and
    // its sum's 4 2^-24 R^2, R a little beyond the cutoff; the band is twice that.
    __device__ __forceinline__ CradTest(const NepDev<double> &P, const Eval2Args<double> &a, int64_t i)
        : pi(a.pos[i]), fi(a.posf[i]) {
        const float u = 5.9604645e-8f;
        const float m = fmaxf(fmaxf(fabsf(fi.x), fabsf(fi.y)), fabsf(fi.z));
        const float L = fmaxf(fmaxf((float)a.box.L[0], (float)a.box.L[1]), (float)a.box.L[2]);
        const float E = u * (8.f * m + 4.f * L + 64.f), Rc = (float)P.rc_r + 1.f;
        band = 2.f * (3.4641017f * Rc * E + 3.f * E * E + 4.f * u * Rc * Rc);
    }
    __device__ __forceinline__ void operator()(const NepDev<double> &P, const Eval2Args<double> &a, int j, const float4 &fj,
                                               bool &in, bool &ang) const {
        float x = fj.x - fi.x, y = fj.y - fi.y, z = fj.z - fi.z;
        minimg(a.boxf, x, y, z);
        const float d2f = x * x + y * y + z * z, r2 = (float)P.rc_r2, a2 = (float)P.rc_a2;
        in = d2f < r2;
        ang = d2f < a2;
        // inside a band (or NaN): the FP64 test decides
        if (!(fabsf(d2f - r2) > band) || !(fabsf(d2f - a2) > band)) {
            double dx, dy, dz;
            sep(a.box, pi, ro(a.pos + j), dx, dy, dz);
            const double d2 = dx * dx + dy * dy + dz * dz;
            in = d2 < P.rc_r2;
            ang = d2 < P.rc_a2;
        }
    }
};

template <typename R>
struct CradSmem {
    R stage[8][CR_STAGE];                // per atom of the block; afterwards its sums [2][5][10]
    R q[CR_NQ][8];                       // the block's descriptor entries, written out by rows
};
struct CradRowsSmem {
    uint32_t mask[MASKW_MAX][8];         // in-cutoff candidate slots of the block's atoms
};
struct CradLists {                       // the one-kernel form: in-cutoff neighbours in list order
    int list[8][32 * MASKW_MAX + 16];    // (padded like the stage)
};

// Where a lane of a wide radial kernel works: 16 lanes per atom, two atoms per warp.
template <typename R>
struct CradPlace {
    int lane, slot8, half, per;   // lane of the atom, atom of the block, its lanes' shift in the warp, atoms per block
    int64_t blk, i, at;           // i: the atom; at: the last one for lanes past it
    bool valid;
    __device__ __forceinline__ CradPlace(const Eval2Args<R> &a, int64_t block)
        : lane(threadIdx.x & (CR_LANES - 1)), slot8(threadIdx.x / CR_LANES), half(threadIdx.x & CR_LANES),
          per(blockDim.x / CR_LANES), blk(block), i(block * (blockDim.x / CR_LANES) + threadIdx.x / CR_LANES),
          at(i < a.n ? i : a.n - 1), valid(i < a.n) {}
};

// A: rows, in-cutoff slots and counts of the atom; list: its in-cutoff neighbours (null: not kept).
// Returns the pairs found, m0 of them of species 0.
template <typename R>
__device__ __forceinline__ int crad_rows(const NepDev<R> &P, const Eval2Args<R> &a, const CradPlace<R> &w,
                                         CradRowsSmem &sm, int *list, int &m0) {
    const int lane = w.lane, half = w.half, slot8 = w.slot8;
    const int64_t N = a.n, i = w.i, at = w.at;
    const unsigned lt = (1u << lane) - 1u;
    if (lane < MASKW_MAX) sm.mask[lane][slot8] = 0u;
    const int4 sg = w.valid ? a.seg[i] : make_int4(0, 0, 0, 0);
    const CradTest<R> test(P, a, at);
    const int32_t *__restrict__ nrow = a.nbr + at * a.capr;
    const uint8_t *__restrict__ rrow = a.rev + at * a.capr;
    __syncwarp();
    int m = 0, na = 0, na0 = 0;   // pairs found, angular ones (of species 0)
    m0 = 0;
    bool ovf = false;
    const int steps = __reduce_max_sync(0xffffffffu, sg.w);
    // the next candidate's FP32 position and the one after it are in flight
    int jn = lane < sg.w ? nrow[lane] : 0, jn2 = lane + CR_LANES < sg.w ? nrow[lane + CR_LANES] : 0;
    float4 pn = a.posf[lane < sg.w ? jn : at];
    uint32_t word = 0u;
    for (int base = 0; base < steps; base += CR_LANES) {
        const int v = base + lane, j = jn;
        const float4 pj = pn;
        jn = jn2;
        if (v + CR_LANES < sg.w) pn = a.posf[jn];
        if (v + 2 * CR_LANES < sg.w) jn2 = nrow[v + 2 * CR_LANES];
        bool in = false, ang = false;
        if (v < sg.w) test(P, a, j, pj, in, ang);
        const unsigned ha = (__ballot_sync(0xffffffffu, ang) >> half) & 0xffffu;
        const int ra = na + __popc(ha & lt);
        if (ang && ra >= a.cap_ang) {   // angular rows full: only after a list overflow
            ovf = true;
            in = ang = false;
        }
        const unsigned hi = (__ballot_sync(0xffffffffu, in) >> half) & 0xffffu;
        if (in) {
            if (list) list[m + __popc(hi & lt)] = j;
            // radial-only pairs are numbered on their own (those kept so far: m - na; of these sixteen: hi
            // without the angular ones), so a refused angular pair leaves no gap in their rows
            const int row = ang ? ra : a.cap_ang + (m - na) + __popc(hi & ~ha & lt);
            stg(a.crow + (int64_t)row * N + i, make_int2(j, rrow[v]));
        }
        word = base & 16 ? word | hi << 16 : hi;
        if (lane == 0) sm.mask[base >> 5][slot8] = word;
        if (base < sg.y) {   // species 0 ends at sg.y
            const unsigned first = base + CR_LANES <= sg.y ? 0xffffu : (1u << (sg.y - base)) - 1u;
            m0 += __popc(hi & first);
            na0 = min(na0 + __popc(ha & first), a.cap_ang);
        }
        m += __popc(hi);
        na = min(na + __popc(ha), a.cap_ang);
    }
    if (ovf) atomicOr(a.status, ST_NBR_OVERFLOW);
    if (w.valid && lane == 0) stg(a.cnt + i, make_int4(na0, na, m0 - na0, m - na));
    __syncwarp();
    return m;
}

// The block's slot masks by words, its descriptor entries by rows: its atoms are neighbours in memory.
template <typename R>
__device__ __forceinline__ void crad_store_masks(const Eval2Args<R> &a, const CradPlace<R> &w, const CradRowsSmem &sm) {
    for (int e = threadIdx.x; e < a.maskw * w.per; e += blockDim.x) {
        const int word = e / w.per, k = e % w.per;
        const int64_t i = w.blk * w.per + k;
        if (i < a.n) stg(reinterpret_cast<int *>(a.mask) + (int64_t)word * a.n + i, (int)sm.mask[word][k]);
    }
}
template <typename R>
__device__ __forceinline__ void crad_store_q(const Eval2Args<R> &a, const CradPlace<R> &w, const CradSmem<R> &sm) {
    for (int e = threadIdx.x; e < CR_NQ * w.per; e += blockDim.x) {
        const int row = e / w.per, k = e % w.per;
        const int64_t i = w.blk * w.per + k;
        const int v = row < 5 ? Q_R + row : row < 25 ? Q_EX + (row - 5) : Q_O;   // EX, DMI, ANI, SIA in turn
        if (i < a.n) stg(a.q + v * a.qs + i, sm.q[row][k]);
    }
}

// B, C: the sums of the atom's m pairs (m0 of species 0 first) and its descriptor entries; neighbour(base): the
// neighbour of the lane's pair of the round from base on.
template <typename R, typename Neighbour>
__device__ __forceinline__ void crad_sums(const NepDev<R> &P, const Eval2Args<R> &a, const CradPlace<R> &w, int m, int m0,
                                          CradSmem<R> &sm, Neighbour neighbour) {
    const int lane = w.lane, slot8 = w.slot8;
    const int64_t at = w.at;
    R *stage = sm.stage[slot8];
    v4<R> pi, si;
    pair_at(a, at, pi, si);
    const int kp = lane % 5, third = lane / 5;   // lane 15 is idle in the sums
    R b0[2][2];
    v2<R> b12[2][2], b34[2][2];
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            b0[t][k] = R(0);
            b12[t][k] = b34[t][k] = pair2<R>(R(0), R(0));
        }
    const int mmax = __reduce_max_sync(0xffffffffu, m);
    for (int base = 0; base < mmax; base += CR_LANES) {
        const int cnt = min(m - base, CR_LANES);
        if (lane < cnt) {
            const int j = neighbour(base);
            v4<R> pj, sj;
            pair_at(a, j, pj, sj);
            R dx, dy, dz;
            sep(a.box, pi, pj, dx, dy, dz);
            const R d2 = dx * dx + dy * dy + dz * dz;
            const R ir = rsqrt_(d2), r = d2 * ir;
            const R ux = dx * ir, uy = dy * ir, uz = dz * ir;
            R f[NK];
            carrier_f(r, P.inv_rc_r, f);
            const R siu = si.x * ux + si.y * uy + si.z * uz;
            const R sju = sj.x * ux + sj.y * uy + sj.z * uz;
            v4<R> *d = reinterpret_cast<v4<R> *>(stage + lane * CR_LD);
            v4<R> w;
            w.x = f[0]; w.y = f[1]; w.z = f[2]; w.w = f[3];
            d[0] = w;
            w.x = f[4]; w.y = f[5]; w.z = f[6]; w.w = f[7];
            d[1] = w;
            v2<R> w2;
            w2.x = f[8]; w2.y = R(0);
            *reinterpret_cast<v2<R> *>(d + 2) = w2;
            w.x = si.x * sj.x + si.y * sj.y + si.z * sj.z;
            w.y = (si.y * sj.z - si.z * sj.y) * ux + (si.z * sj.x - si.x * sj.z) * uy + (si.x * sj.y - si.y * sj.x) * uz;
            w.z = siu * sju;
            w.w = siu * siu;
            d[3] = w;
        }
        __syncwarp();
        const int split = min(max(m0 - base, 0), max(cnt, 0));   // staged pairs of species 0
        if (third < 3) {
            auto add = [&](int t, int x) {
                const v2<R> f = *reinterpret_cast<const v2<R> *>(stage + x * CR_LD + 2 * kp);
                const v4<R> g = *reinterpret_cast<const v4<R> *>(stage + x * CR_LD + 12);
                b0[t][0] += f.x;
                b0[t][1] += f.y;
                b12[t][0] = fma2(pair2<R>(f.x, f.x), pair2<R>(g.x, g.y), b12[t][0]);
                b34[t][0] = fma2(pair2<R>(f.x, f.x), pair2<R>(g.z, g.w), b34[t][0]);
                b12[t][1] = fma2(pair2<R>(f.y, f.y), pair2<R>(g.x, g.y), b12[t][1]);
                b34[t][1] = fma2(pair2<R>(f.y, f.y), pair2<R>(g.z, g.w), b34[t][1]);
            };
            for (int x = third; x < split; x += 3) add(0, x);
            for (int x = split + third; x < cnt; x += 3) add(1, x);
        }
        __syncwarp();
    }
    // C: the three thirds, then q = sum over species and k
    R *sums = stage;   // [species][group][10]
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        R v[5][2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            v[0][k] = b0[t][k];
            v[1][k] = b12[t][k].x;
            v[2][k] = b12[t][k].y;
            v[3][k] = b34[t][k].x;
            v[4][k] = b34[t][k].y;
        }
#pragma unroll
        for (int g = 0; g < 5; ++g) {
            v2<R> s;
            s.x = v[g][0] + __shfl_down_sync(0xffffffffu, v[g][0], 5, CR_LANES) +
                  __shfl_down_sync(0xffffffffu, v[g][0], 10, CR_LANES);
            s.y = v[g][1] + __shfl_down_sync(0xffffffffu, v[g][1], 5, CR_LANES) +
                  __shfl_down_sync(0xffffffffu, v[g][1], 10, CR_LANES);
            if (lane < 5) *reinterpret_cast<v2<R> *>(sums + (t * 5 + g) * 10 + 2 * kp) = s;
        }
    }
    __syncwarp();
    const R *__restrict__ ct = a.ctab + (at < a.n_fe ? 0 : 1) * (2 * NK * 32);
    for (int o = lane; o < 25; o += CR_LANES) {
        const int g = o / NCH;
        R q = R(0);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const v2<R> *s = reinterpret_cast<const v2<R> *>(sums + (t * 5 + g) * 10);
#pragma unroll
            for (int k = 0; k < NK; k += 2) {
                const v2<R> x = s[k / 2];
                q += ro(ct + (t * NK + k) * 32 + o) * x.x;
                if (k + 1 < NK) q += ro(ct + (t * NK + k + 1) * 32 + o) * x.y;
            }
        }
        sm.q[o][slot8] = q;
    }
    if (lane == 0) sm.q[25][slot8] = si.x * si.x + si.y * si.y + si.z * si.z;
}

// In one kernel.
template <typename R>
__device__ __forceinline__ void crad_wide_body(const NepDev<R> &P, const Eval2Args<R> &args, int64_t blk,
                                               CradSmem<R> &sm, CradRowsSmem &rows, CradLists &lists) {
    // the arguments as values: read once from the block's copy, so nothing in the loops below
    // depends on where they are stored
    const Eval2Args<R> a = args;
    if (a.split || (a.skip && *a.skip)) return;
    const CradPlace<R> w(a, blk);
    int *list = lists.list[w.slot8], m0;
    const int m = crad_rows(P, a, w, rows, list, m0);
    crad_sums(P, a, w, m, m0, sm, [&](int base) { return list[base + w.lane]; });
    __syncthreads();
    crad_store_masks(a, w, rows);
    crad_store_q(a, w, sm);
}

// In two (crad_is_split): the rows, then the sums over them, which nothing before the network waits for and which
// run beside the angular kernel, where a small system leaves both most of the GPU.  A step of 512 / 1,728 /
// 4,096 / 8,000 / 13,824 atoms, mixed precision: 44.4 / 49.7 / 58.6 / 71.4 / 101.2 us in one kernel, 40.9 / 46.7 / 56.5 / 72.8 /
// 104.5 in two; FP64, 512 / 1,728 / 2,744 / 4,096 atoms: 185 / 373 / 571 / 641 and 173 / 377 / 554 / 692 us.  (The line
// lies below where the two cross.)
template <typename R>
__device__ __forceinline__ void crad_rows_body(const NepDev<R> &P, const Eval2Args<R> &args, int64_t blk, CradRowsSmem &sm) {
    const Eval2Args<R> a = args;
    if (!a.split || (a.skip && *a.skip)) return;
    const CradPlace<R> w(a, blk);
    int m0;
    crad_rows(P, a, w, sm, nullptr, m0);
    __syncthreads();
    crad_store_masks(a, w, sm);
}
template <typename R>
__device__ __forceinline__ void crad_sums_body(const NepDev<R> &P, const Eval2Args<R> &args, int64_t blk, CradSmem<R> &sm) {
    const Eval2Args<R> a = args;
    if (!a.split || (a.skip && *a.skip)) return;
    const CradPlace<R> w(a, blk);
    // pairs by species, angular rows before the others; the next round's neighbour is in flight
    const int4 c = w.valid ? a.cnt[w.i] : make_int4(0, 0, 0, 0);   // angular of species 0, angular, others of species 0, others
    const int m = c.y + c.w, m0 = c.x + c.z;
    auto row = [&](int p) {
        if (p < m0) return p < c.x ? p : a.cap_ang + p - c.x;
        const int r = p - m0 + c.x;
        return r < c.y ? r : a.cap_ang + c.z + (r - c.y);
    };
    const int2 *__restrict__ crow = a.crow + w.at;
    int jn = w.lane < m ? crow[(int64_t)row(w.lane) * a.n].x : 0;
    crad_sums(P, a, w, m, m0, sm, [&](int base) {
        const int j = jn, p = base + CR_LANES + w.lane;
        if (p < m) jn = crow[(int64_t)row(p) * a.n].x;
        return j;
    });
    __syncthreads();
    crad_store_q(a, w, sm);
}


// ------------------------------------------------------------------ k_ang_fwd
// LPA lanes per atom (4, or 32 in small systems: eval_is_wide): each stages one pair, then each takes the harmonics
// of lm_of.  Stage of one angular pair: (g_n, s g_n) interleaved for n = 0..4, pad (2),
// then the 24 harmonics in lane-major order, so each lane reads its own from consecutive places (four
// lanes: the first four of each lane's six, then the last two of each).
constexpr int FSTAGE = 36;
constexpr int FWARP = 32 * FSTAGE + 20;   // a warp's stages
template <int LPA>
struct AngLanes {
    static constexpr int H = (NLM + LPA - 1) / LPA;     // harmonics per lane
    static_assert(LPA == 4 || LPA == 32, "24 harmonics in equal shares, or one per lane");
    // harmonic at place t of a stage
    static constexpr __device__ int lm_at(int t) {
        if (LPA == 32) return t;
        return t < 16 ? lm_of<4>(t / 4, t % 4) : lm_of<4>((t - 16) / 2, 4 + t % 2);
    }
    // Atom grp's stages in its warp's.  With four lanes per atom (FP32) the eight atoms start in different
    // groups of four banks, 16 banks apart within a pair of atoms and 8 between pairs, so that eight
    // lanes writing their stages, a quad reading one together and the lanes reading their own
    // harmonics meet no bank twice.  What bounds the kernel is the shared-memory and L1 data path (59%
    // busy, issue 56%); with the quads 4 words apart (74% busy) a third of the shared-memory wavefronts were
    // bank conflicts: 519 to 493 us at 884,736 atoms, 79 to 75 us at 110,592.
    static __device__ int stage_at(int grp) {
        return LPA == 32 ? 0 : grp * (4 * FSTAGE) + 8 * ((grp >> 1) & 1) + 12 * (grp >> 2);
    }
};

// g_n of the angular channels and the harmonics at u.  FP64, bound by its pipe: the contraction without
// the f_k (see Carrier) and the harmonics from shared products, some 25 of 150 FP64 instructions of a
// staged pair less (1,719 to 1,652 us at 110,592 atoms); FP32, which the shared-memory path
// bounds, gains nothing from either (518 to 520 us at 884,736 atoms).
template <typename R, int TI, int TJ>
__device__ __forceinline__ void ang_g(const NepDev<R> &P, R r, R inv_rc, R g[NCH]) {
    if constexpr (sizeof(R) == 4) {
        R f[NK];
        carrier_f(r, inv_rc, f);
        contract_k<R, TI, TJ, G_A>(P, f, g);
    } else {
        const R t = r * inv_rc, fch = cut_half(t), y = t - R(1), x = fma_(R(2) * y, y, R(-1)), x2 = R(2) * x;
        R pn[NCH], m = R(1), c = x;
#pragma unroll
        for (int n = 0; n < NCH; ++n) pn[n] = fma_(P.c[TI][TJ][G_A][n][1], x, P.ca0[TI][TJ][n]);
#pragma unroll
        for (int k = 2; k < NK; ++k) {
            const R tk = fma_(x2, c, -m);
#pragma unroll
            for (int n = 0; n < NCH; ++n) pn[n] = fma_(P.c[TI][TJ][G_A][n][k], tk, pn[n]);
            m = c;
            c = tk;
        }
#pragma unroll
        for (int n = 0; n < NCH; ++n) g[n] = fch * pn[n];
    }
}
__device__ __forceinline__ void ang_harm(float x, float y, float z, float p[NLM]) { harm_p(x, y, z, p); }
__device__ __forceinline__ void ang_harm(double x, double y, double z, double p[NLM]) {
    const double x2 = x * x, y2 = y * y, z2 = z * z, q = x2 + y2, r2 = q + z2;
    const double xy = x * y, yz = y * z, xz = x * z, d = x2 - y2;
    const double c1 = fma(3.0, x2, -y2), c2 = fma(-3.0, y2, x2), c3 = fma(4.0, z2, -q);
    const double c5 = fma(6.0, z2, -q), c6 = fma(4.0, z2, -3.0 * q);
    p[0] = x; p[1] = y; p[2] = z;
    p[3] = xy; p[4] = yz; p[5] = xz; p[6] = d; p[7] = fma(2.0, z2, -q);
    p[8] = y * c1; p[9] = xy * z; p[10] = y * c3; p[11] = z * fma(2.0, z2, -3.0 * q); p[12] = x * c3; p[13] = z * d;
    p[14] = x * c2;
    p[15] = xy * d; p[16] = yz * c1; p[17] = xy * c5; p[18] = yz * c6;
    p[19] = fma(z2, fma(35.0, z2, -30.0 * r2), 3.0 * r2 * r2);
    p[20] = xz * c6; p[21] = d * c5; p[22] = xz * c2; p[23] = fma(d, d, -4.0 * xy * xy);
}

template <typename R, int LPA, int TI, int TJ>
__device__ __forceinline__ void ang_stage_fwd(const NepDev<R> &P, const Eval2Args<R> &a, const v4<R> &pi,
                                              const v4<R> &si, const v4<R> &pj, const v4<R> &sj, R *st) {
    R dx, dy, dz;
    sep(a.box, pi, pj, dx, dy, dz);
    const R d2 = dx * dx + dy * dy + dz * dz;
    const R ir = rsqrt_(d2), r = d2 * ir;
    R g[NCH];
    ang_g<R, TI, TJ>(P, r, P.inv_rc_a, g);
    const R s = si.x * sj.x + si.y * sj.y + si.z * sj.z;
    v4<R> w0, w1;
    v2<R> w2;
    w0.x = g[0]; w0.y = g[0] * s; w0.z = g[1]; w0.w = g[1] * s;
    w1.x = g[2]; w1.y = g[2] * s; w1.z = g[3]; w1.w = g[3] * s;
    w2.x = g[4]; w2.y = g[4] * s;
    reinterpret_cast<v4<R> *>(st)[0] = w0;
    reinterpret_cast<v4<R> *>(st)[1] = w1;
    reinterpret_cast<v2<R> *>(st)[4] = w2;
    R p[NLM];
    ang_harm(dx * ir, dy * ir, dz * ir, p);
    using L = AngLanes<LPA>;
#pragma unroll
    for (int t = 0; t < NLM; t += 2) reinterpret_cast<v2<R> *>(st)[6 + t / 2] = pair2<R>(p[L::lm_at(t)], p[L::lm_at(t + 1)]);
}

template <typename R, int LPA>
__device__ __forceinline__ void ang_fwd_body(const NepDev<R> &P, const Eval2Args<R> &args, int64_t blk,
                                             unsigned char *smem_raw) {
    // the arguments as values: read once from the block's copy, so nothing in the loops below
    // depends on where they are stored
    const Eval2Args<R> a = args;
    if (a.skip && *a.skip) return;
    using L = AngLanes<LPA>;
    constexpr int H = L::H, APW = 32 / LPA;   // harmonics per lane, atoms per warp
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = lane / LPA, ql = lane % LPA;
    const int64_t i = (blk * (blockDim.x >> 5) + warp) * APW + grp;
    const bool valid = i < a.n;
    R *stage = reinterpret_cast<R *>(smem_raw) + warp * FWARP + L::stage_at(grp);
    v4<R> pi, si;
    int na0 = 0, na = 0, ti = 0;
    if (valid) {
        pair_at(a, i, pi, si);
        const int4 c = a.cnt[i];
        na0 = c.x;
        na = c.y;
        ti = i < a.n_fe ? 0 : 1;
    }
    v2<R> BB[H][NCH];   // (B_nlm, BS_nlm) of the lane's harmonics
#pragma unroll
    for (int m = 0; m < H; ++m)
#pragma unroll
        for (int n = 0; n < NCH; ++n) BB[m][n] = pair2<R>(R(0), R(0));
    const int nmax = __reduce_max_sync(0xffffffffu, na);
    // the lane's list entry three rounds ahead and its coordinates two rounds ahead are in flight
    v4<R> pjn, sjn, pjn2, sjn2;
    int jn3 = 0;
    const int2 *__restrict__ crow = a.crow + i;
    const int64_t N = a.n;
    if (ql < na) {
        const int j = crow[(int64_t)ql * N].x;
        pair_at(a, j, pjn, sjn);
    }
    if (ql + LPA < na) {
        const int j = crow[(int64_t)(ql + LPA) * N].x;
        pair_at(a, j, pjn2, sjn2);
    }
    if (ql + 2 * LPA < na) jn3 = crow[(int64_t)(ql + 2 * LPA) * N].x;
    for (int base = 0; base < nmax; base += LPA) {
        const int p = base + ql;
        const v4<R> pj = pjn, sj = sjn;
        pjn = pjn2;
        sjn = sjn2;
        if (p + 2 * LPA < na) {
            pair_at(a, jn3, pjn2, sjn2);
        }
        if (p + 3 * LPA < na) jn3 = crow[(int64_t)(p + 3 * LPA) * N].x;
        if (p < na) {
            R *st = stage + ql * FSTAGE;
            if (ti == 0) {
                if (p < na0) ang_stage_fwd<R, LPA, 0, 0>(P, a, pi, si, pj, sj, st);
                else ang_stage_fwd<R, LPA, 0, 1>(P, a, pi, si, pj, sj, st);
            } else {
                if (p < na0) ang_stage_fwd<R, LPA, 1, 0>(P, a, pi, si, pj, sj, st);
                else ang_stage_fwd<R, LPA, 1, 1>(P, a, pi, si, pj, sj, st);
            }
        }
        __syncwarp();
        const int cnt = LPA * H > NLM && ql >= NLM ? 0 : min(LPA, na - base);   // lanes without a harmonic
        for (int q = 0; q < cnt; ++q) {
            const R *sp = stage + q * FSTAGE;
            const v4<R> w0 = reinterpret_cast<const v4<R> *>(sp)[0];
            const v4<R> w1 = reinterpret_cast<const v4<R> *>(sp)[1];
            const v2<R> w2 = reinterpret_cast<const v2<R> *>(sp)[4];
            const v2<R> gg[NCH] = {pair2<R>(w0.x, w0.y), pair2<R>(w0.z, w0.w), pair2<R>(w1.x, w1.y),
                                   pair2<R>(w1.z, w1.w), w2};
            R pv[H];
            if constexpr (LPA == 4) {
                const v4<R> x = *reinterpret_cast<const v4<R> *>(sp + 12 + 4 * ql);
                const v2<R> y = *reinterpret_cast<const v2<R> *>(sp + 28 + 2 * ql);
                pv[0] = x.x; pv[1] = x.y; pv[2] = x.z; pv[3] = x.w; pv[4] = y.x; pv[5] = y.y;
            } else {
#pragma unroll
                for (int m = 0; m < H; ++m) pv[m] = sp[12 + H * ql + m];
            }
#pragma unroll
            for (int m = 0; m < H; ++m) {
                const v2<R> pl = pair2<R>(pv[m], pv[m]);
#pragma unroll
                for (int n = 0; n < NCH; ++n) BB[m][n] = fma2(gg[n], pl, BB[m][n]);
            }
        }
        __syncwarp();
    }
    // angular sums for the backward pass, and the channel values: with four lanes per atom summed in
    // registers and over the quad, else through the atom's stage
    constexpr bool QUAD = LPA == 4;
    [[maybe_unused]] R qa[QUAD ? NCH : 1][4], qs[QUAD ? NCH : 1][4];
    if constexpr (QUAD) {
#pragma unroll
        for (int n = 0; n < NCH; ++n)
#pragma unroll
            for (int l = 0; l < 4; ++l) { qa[n][l] = R(0); qs[n][l] = R(0); }
    }
#pragma unroll
    for (int m = 0; m < H; ++m) {
        const int lm = lm_of<LPA>(ql, m);
        if (!QUAD && lm >= NLM) break;
        const int l = l_of_lm(lm) - 1;
        const R kap = kappa_of_lm<R>(lm);
        if (valid) {   // the harmonic's record: (B_n, BS_n) for n = 0..4; two harmonics' in five pieces
            R *rec = a.bsum + ((int64_t)i * NLM + lm) * BREC;
            if constexpr (!QUAD) {
#pragma unroll
                for (int n = 0; n < NCH; ++n) stg(reinterpret_cast<v2<R> *>(rec) + n, BB[m][n]);
            } else if (m % 2 == 0) {
                const v2<R> *p = BB[m], *q = BB[m + (H > 1 ? 1 : 0)];
                v4<R> *rec4 = reinterpret_cast<v4<R> *>(rec);
                stg(rec4, quad4<R>(p[0], p[1])); stg(rec4 + 1, quad4<R>(p[2], p[3])); stg(rec4 + 2, quad4<R>(p[4], q[0]));
                stg(rec4 + 3, quad4<R>(q[1], q[2])); stg(rec4 + 4, quad4<R>(q[3], q[4]));
            }
        }
#pragma unroll
        for (int n = 0; n < NCH; ++n) {
            const R Bv = BB[m][n].x, BSv = BB[m][n].y;
            const R ka = kap * Bv * Bv, ks = kap * BSv * BSv;
            if constexpr (QUAD) {
                // l is 1..4 depending on the lane: add into the matching slot
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    qa[n][t] += (t == l) ? ka : R(0);
                    qs[n][t] += (t == l) ? ks : R(0);
                }
            } else {   // [lm][2 n + (0: A, 1: SA)]
                *reinterpret_cast<v2<R> *>(stage + lm * 10 + 2 * n) = pair2<R>(ka, ks);
            }
        }
    }
    if constexpr (QUAD) {
        // summed over the quad, lane ql ending with l = ql + 1: the pair of lanes that differ in bit 0
        // exchange the degrees the other keeps, then those that differ in bit 1
        const bool odd = ql & 1, high = ql & 2;
#pragma unroll
        for (int n = 0; n < NCH; ++n) {
            R v[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const R *x = c == 0 ? qa[n] : qs[n];
                const R lo = (odd ? x[1] : x[0]) + __shfl_xor_sync(0xffffffffu, odd ? x[0] : x[1], 1);
                const R hi = (odd ? x[3] : x[2]) + __shfl_xor_sync(0xffffffffu, odd ? x[2] : x[3], 1);
                v[c] = (high ? hi : lo) + __shfl_xor_sync(0xffffffffu, high ? lo : hi, 2);
            }
            if (valid) {
                stg(a.q + (int64_t)(Q_A + n * 4 + ql) * a.qs + i, v[0]);
                stg(a.q + (int64_t)(Q_SA + n * 4 + ql) * a.qs + i, v[1]);
            }
        }
    } else {
        __syncwarp();
        if (valid) {   // the lanes take the 40 values
            for (int o = ql; o < 8 * NCH; o += LPA) {
                const int l = o & 3, c = o >> 2;   // c: 2 n + (0: A, 1: SA)
                R v = R(0);
                for (int lm = l * (l + 2); lm < (l + 1) * (l + 3); ++lm) v += stage[lm * 10 + c];
                stg(a.q + (int64_t)((c & 1 ? Q_SA : Q_A) + (c >> 1) * 4 + l) * a.qs + i, v);
            }
        }
    }
}


// ------------------------------------------------------------------ k_bwd (fused)
// Quad per atom, lanes over pairs.  Shared memory per atom: the angular adjoints
// dE/dB_nlm, dE/dBS_nlm as 24 records of 10 ((dE/dB, dE/dBS) interleaved per n), then the precontracted
// radial coefficients C^G_k = sum_n Fp^G_n c^G_{n k t_i t_j} for both neighbour
// species (2 x 48).  336 mod 32 = 16 and four words more every second atom: the eight atoms of a warp
// read disjoint groups of four banks, and two atoms' lanes storing their records meet no bank twice.
// What bounds the FP32 kernel is its loads, of which the records' (60 16-byte words an angular pair)
// are most of the shared-memory ones: without the two pads a 12-word record had, the backward at
// 884,736 atoms takes 1.49 instead of 1.55 ms and the angular kernel, which writes them, 483 instead of
// 493 us (110,592: 220 / 73.5 instead of 227 / 75 us; FP64 unchanged).
constexpr int BW_C = NLM * BREC;
constexpr int BW_ATOM = BW_C + 96;
constexpr int BW_WARP = 8 * BW_ATOM + 16;
template <int LPA>
__device__ __forceinline__ int bwd_at(int grp) { return LPA == 4 ? grp * BW_ATOM + 4 * (grp >> 1) : 0; }

template <typename R>
struct BwdAcc2 {
    R fx, fy, fz, hx, hy, hz;
    R w[9];
};

// The atom's precontracted radial coefficients C^G_k = sum_n Fp^G_n c^G_nk for both neighbour species
// into smc, 48 each: [k][EX, DMI, ANI, SIA], then R by k.  Lane ql of four takes group ql of the four
// magnetic ones (fm: its five gradient entries) and k = 2 ql, 2 ql + 1 of group R (fr), lane 0 also R's
// k = 8, from the centre's rows ct of the table; species tj0 .. tj0 + NT - 1.  (FP32 had every lane form
// all 90 from constant operands, and every lane fetch the entries of its own harmonics: with the
// shares here and the entries handed round through shared memory the backward at 884,736 atoms takes
// 1.55 instead of 1.69 ms, at 110,592 227 instead of 248 us, with a warp per atom at 512 12.5 instead of
// 14.0 us.  Fetching the entries' records with asynchronous copies instead: 1.62 ms.)
constexpr int BW_CR = 4 * NK;   // group R's place
__device__ __forceinline__ constexpr int coeff_at(int g, int k) { return g == 0 ? BW_CR + k : 4 * k + g - 1; }
template <typename R, int NT>
__device__ __forceinline__ void bwd_coeffs(const R *__restrict__ ct, const R fm[NCH], const R fr[NCH], int ql, int tj0,
                                           R *smc) {
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        const R *__restrict__ row = ct + (tj0 + t) * (NCH * 5 * CB_ROW);
        v2<R> c[4], cr = pair2<R>(R(0), R(0));
        R c8 = R(0), cr8 = R(0);
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] = pair2<R>(R(0), R(0));
#pragma unroll
        for (int n = 0; n < NCH; ++n, row += 5 * CB_ROW) {
            const R *m = row + ql * CB_ROW, *r = row + 4 * CB_ROW;
            const v4<R> a = *reinterpret_cast<const v4<R> *>(m), b = *reinterpret_cast<const v4<R> *>(m + 4);
            const v2<R> f2 = pair2<R>(fm[n], fm[n]);
            c[0] = fma2(f2, pair2<R>(a.x, a.y), c[0]);
            c[1] = fma2(f2, pair2<R>(a.z, a.w), c[1]);
            c[2] = fma2(f2, pair2<R>(b.x, b.y), c[2]);
            c[3] = fma2(f2, pair2<R>(b.z, b.w), c[3]);
            c8 = fma_(fm[n], m[8], c8);
            cr = fma2(pair2<R>(fr[n], fr[n]), *reinterpret_cast<const v2<R> *>(r + 2 * ql), cr);
            cr8 = fma_(fr[n], r[8], cr8);
        }
        R *d = smc + (tj0 + t) * 48;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            d[8 * q + ql] = c[q].x;
            d[8 * q + 4 + ql] = c[q].y;
        }
        d[32 + ql] = c8;
        *reinterpret_cast<v2<R> *>(d + BW_CR + 2 * ql) = cr;
        if (ql == 0) d[BW_CR + 8] = cr8;
    }
}

// g_n and dg_n/dr of the angular channels
template <typename R, int TI, int TJ>
__device__ __forceinline__ void ang_gdg(const NepDev<R> &P, R r, R inv_rc, R g[NCH], R dg[NCH]) {
    if constexpr (sizeof(R) == 4) {
        R f[NK], df[NK];
        carrier_fd2(r, inv_rc, f, df);
        contract_k2<R, TI, TJ, G_A>(P, f, df, g, dg);
        return;
    }
    const Carrier<R> cr(r, inv_rc);
    v2<R> pq[NCH];
#pragma unroll
    for (int n = 0; n < NCH; ++n) {
        const R c1 = P.c[TI][TJ][G_A][n][1];
        pq[n] = pair2<R>(fma_(c1, cr.x, P.ca0[TI][TJ][n]), c1);
    }
    cr.terms([&](int k, const v2<R> &td) {
#pragma unroll
        for (int n = 0; n < NCH; ++n) {
            const R c = P.c[TI][TJ][G_A][n][k];
            pq[n] = fma2(pair2<R>(c, c), td, pq[n]);
        }
    });
#pragma unroll
    for (int n = 0; n < NCH; ++n) {
        g[n] = cr.fch * pq[n].x;
        dg[n] = fma_(cr.dxf, pq[n].y, cr.dfch * pq[n].x);
    }
}

// The angular adjoint of one pair from the atom's adjoint records bb[lm] = (dE/dB_n, dE/dBS_n) and
// the harmonics p_lm at u.  With a_lm = sum_n g_n (dE/dB + s dE/dBS) the chain rule gives
//   dE/dr along u    sum_lm p_lm sum_n g_n' (dE/dB + s dE/dBS)
//   dE/du            sum_lm a_lm grad p_lm, of which only the part across u counts
//   dE/ds            sum_lm p_lm sum_n g_n dE/dBS
// and u . grad p_lm = l p_lm, so the part along u is taken out of the vector sum once, by its
// projection, instead of harmonic by harmonic.
//
// FP32: harmonic by harmonic (few values live at a time; the backward at 884,736 atoms 1.62 to 1.58 ms
// against subtracting each harmonic's part along u).
template <typename R, int LM>
__device__ __forceinline__ void bwd_harm(const R *__restrict__ bb, R ux, R uy, R uz, R s, const R g[NCH],
                                         const R dg[NCH], v2<R> &along, R &avx, R &avy, R &avz, R &cj, v4<R> &mid) {
    R p, gx, gy, gz;
    harm_one<R, LM>(ux, uy, uz, p, gx, gy, gz);
    // (dE/dB_n, dE/dBS_n); the records of harmonics 2 k and 2 k + 1 are five 16-byte pieces
    const v4<R> *rec = reinterpret_cast<const v4<R> *>(bb + BREC * (LM & ~1));
    v2<R> Bp[NCH];
    if constexpr (LM % 2 == 0) {
        const v4<R> r0 = rec[0], r1 = rec[1];
        mid = rec[2];
        Bp[0] = pair2<R>(r0.x, r0.y); Bp[1] = pair2<R>(r0.z, r0.w); Bp[2] = pair2<R>(r1.x, r1.y);
        Bp[3] = pair2<R>(r1.z, r1.w); Bp[4] = pair2<R>(mid.x, mid.y);
    } else {
        const v4<R> r3 = rec[3], r4 = rec[4];
        Bp[0] = pair2<R>(mid.z, mid.w); Bp[1] = pair2<R>(r3.x, r3.y); Bp[2] = pair2<R>(r3.z, r3.w);
        Bp[3] = pair2<R>(r4.x, r4.y); Bp[4] = pair2<R>(r4.z, r4.w);
    }
    v2<R> aa = pair2<R>(R(0), R(0)), bq = pair2<R>(R(0), R(0));
#pragma unroll
    for (int n = 0; n < NCH; ++n) {
        aa = fma2(Bp[n], pair2<R>(g[n], g[n]), aa);
        bq = fma2(Bp[n], pair2<R>(dg[n], dg[n]), bq);
    }
    const R av = aa.x + s * aa.y;
    along = fma2(bq, pair2<R>(p, p), along);
    avx += av * gx;
    avy += av * gy;
    avz += av * gz;
    cj += aa.y * p;
    if constexpr (LM + 1 < NLM) bwd_harm<R, LM + 1>(bb, ux, uy, uz, s, g, dg, along, avx, avy, avz, cj, mid);
}

// FP64, where instructions count and registers do not: the sums over n and lm are exchanged,
//   Psi_n = sum_lm p_lm (dE/dB_n, dE/dBS_n), along u sum_n g_n' Psi_n, dE/ds sum_n g_n Psi^S_n,
// and the gradient of a solid harmonic being a combination of those one degree lower, sum_lm a_lm
// grad p_lm is formed from the p of degree l - 1 and a few sums of a's.  With Carrier this takes an
// angular pair from some 1,040 to 780 FP64 instructions: the backward at 110,592 atoms 7.59 to
// 6.41 ms.
template <typename R>
struct AngAdjoint {
    const R *bb;
    R s;
    const R *g;
    v2<R> psi[NCH];
    // harmonic lm = value p: Psi_n advanced, a_lm returned
    __device__ __forceinline__ R take(int lm, R p) {
        const v2<R> *rec = reinterpret_cast<const v2<R> *>(bb + BREC * lm);
        const v2<R> Bp[NCH] = {rec[0], rec[1], rec[2], rec[3], rec[4]};
        v2<R> aa = pair2<R>(Bp[0].x * g[0], Bp[0].y * g[0]);
#pragma unroll
        for (int n = 1; n < NCH; ++n) aa = fma2(Bp[n], pair2<R>(g[n], g[n]), aa);
#pragma unroll
        for (int n = 0; n < NCH; ++n) psi[n] = fma2(Bp[n], pair2<R>(p, p), psi[n]);
        return fma_(s, aa.y, aa.x);
    }
};

template <typename R>
__device__ __forceinline__ void bwd_angular(const R *__restrict__ bb, R x, R y, R z, R s, const R g[NCH],
                                            const R dg[NCH], R &along, R &vx, R &vy, R &vz, R &cj) {
    AngAdjoint<R> A;
    A.bb = bb;
    A.s = s;
    A.g = g;
#pragma unroll
    for (int n = 0; n < NCH; ++n) A.psi[n] = pair2<R>(R(0), R(0));
    // degree 1
    vx = A.take(0, x);
    vy = A.take(1, y);
    vz = A.take(2, z);
    // degree 2: xy, yz, xz, x^2 - y^2, 2 z^2 - x^2 - y^2
    const R x2 = x * x, y2 = y * y, z2 = z * z, q = x2 + y2;
    const R p3 = x * y, p4 = y * z, p5 = x * z, p6 = x2 - y2, p7 = fma_(R(2), z2, -q);
    {
        const R a3 = A.take(3, p3), a4 = A.take(4, p4), a5 = A.take(5, p5), a6 = A.take(6, p6), a7 = A.take(7, p7);
        vx += a3 * y + a5 * z + R(2) * (a6 - a7) * x;
        vy += a3 * x + a4 * z - R(2) * (a6 + a7) * y;
        vz += a4 * y + a5 * x + R(4) * a7 * z;
    }
    // degree 3
    const R c1 = fma_(R(3), x2, -y2), c2 = fma_(R(-3), y2, x2), c3 = fma_(R(4), z2, -q);
    const R p8 = y * c1, p9 = p3 * z, p10 = y * c3, p11 = z * fma_(R(2), z2, R(-3) * q), p12 = x * c3, p13 = z * p6,
            p14 = x * c2;
    {
        const R a8 = A.take(8, p8), a9 = A.take(9, p9), a10 = A.take(10, p10), a11 = A.take(11, p11),
                a12 = A.take(12, p12), a13 = A.take(13, p13), a14 = A.take(14, p14);
        const R d11 = R(6) * a11, d10 = R(2) * a10, d12 = R(2) * a12;
        vx += p3 * fma_(R(6), a8, -d10) + p4 * a9 + p5 * fma_(R(2), a13, -d11) + p6 * fma_(R(3), a14, -a12) + p7 * d12;
        vy += p3 * fma_(R(-6), a14, -d12) + p4 * fma_(R(-2), a13, -d11) + p5 * a9 + p6 * fma_(R(3), a8, a10) + p7 * d10;
        vz += p3 * a9 + R(4) * (p4 * d10 + p5 * d12) + p6 * a13 + R(0.5) * p7 * d11;
    }
    // degree 4
    {
        const R c5 = fma_(R(6), z2, -q), c6 = fma_(R(4), z2, R(-3) * q), r2 = q + z2;
        const R a15 = A.take(15, p3 * p6), a16 = A.take(16, p4 * c1), a17 = A.take(17, p3 * c5),
                a18 = A.take(18, p4 * c6),
                a19 = A.take(19, fma_(z2, fma_(R(35), z2, R(-30) * r2), R(3) * r2 * r2)),
                a20 = A.take(20, p5 * c6), a21 = A.take(21, p6 * c5), a22 = A.take(22, p5 * c2),
                a23 = A.take(23, fma_(p6, p6, R(-4) * p3 * p3));
        const R e17 = R(0.5) * a17, d17 = R(1.5) * a17, d19 = R(12) * a19, d21 = R(3) * a21;
        vx += p8 * (a15 - e17) + p9 * (R(6) * (a16 - a18)) + p10 * d17 + p11 * (R(2) * a20) + p12 * (d21 - d19) +
              p13 * (R(3) * (a22 - a20)) + p14 * fma_(R(4), a23, -a21);
        vy += p14 * (a15 + e17) - p9 * (R(6) * (a20 + a22)) + p12 * d17 + p11 * (R(2) * a18) - p10 * (d21 + d19) +
              p13 * (R(3) * (a16 + a18)) - p8 * fma_(R(4), a23, a21);
        vz += p8 * a16 + p14 * a22 + R(8) * p9 * d17 + R(3) * (p10 * a18 + p12 * a20) + R(16) * p11 * a19 +
              R(4) * p13 * d21;
    }
    v2<R> b = pair2<R>(R(0), R(0));
    cj = R(0);
#pragma unroll
    for (int n = 0; n < NCH; ++n) {
        b = fma2(A.psi[n], pair2<R>(dg[n], dg[n]), b);
        cj = fma_(g[n], A.psi[n].y, cj);
    }
    along = fma_(s, b.y, b.x);
}

// one pair record: FP32 as a single 256-bit store (the record is one 32-byte sector), FP64 as
// two 32-byte stores
__device__ __forceinline__ void store_rec(PairRec<float> *p, const float4 &a, const float4 &b) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
                 "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}
__device__ __forceinline__ void store_rec(PairRec<double> *p, const double4 &a, const double4 &b) {
    stg(&p->a, a);
    stg(&p->b, b);
}

// VIR: the evaluation accumulates the virial parts (a compile-time switch, so the step's
// evaluation keeps no virial accumulators live across its row loops)
template <typename R, bool ANG, bool VIR>
__device__ __forceinline__ void bwd_pair(const NepDev<R> &P, const Eval2Args<R> &a, int ti, int tj, const v4<R> &pi,
                                         const v4<R> &si, const v4<R> &pj, const v4<R> &sj, int j, int t,
                                         const R *sm, BwdAcc2<R> &acc) {
    R dx, dy, dz;
    sep(a.box, pi, pj, dx, dy, dz);
    const R d2 = dx * dx + dy * dy + dz * dz;
    const R ir = rsqrt_(d2), r = d2 * ir;
    const R ux = dx * ir, uy = dy * ir, uz = dz * ir;
    // radial and pairwise-magnetic part with the precontracted coefficients: the values h of the
    // four magnetic groups, then the slope along the pair of every group's term together.  (The
    // carrier comes before the coefficients' loads and the spin products after the contraction:
    // held across it they cost FP32 the registers of its prefetch, 1.62 instead of 1.58 ms.)
    R C[48];
    auto load_coefficients = [&]() {
        const v4<R> *cv = reinterpret_cast<const v4<R> *>(sm + BW_C + tj * 48);
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            const v4<R> c4 = cv[q];
            C[4 * q] = c4.x; C[4 * q + 1] = c4.y; C[4 * q + 2] = c4.z; C[4 * q + 3] = c4.w;
        }
    };
    [[maybe_unused]] v2<R> pq[5];         // FP64: (P, Q) per group
    [[maybe_unused]] R e0 = 0, dfch = 0, dxf = 0;
    [[maybe_unused]] v2<R> he[4];         // FP32: (h_G, e_G) of the four magnetic groups
    R h1, h2, h3, h4;
    if constexpr (sizeof(R) == 8) {
        const Carrier<R> cr(r, P.inv_rc_r);
        load_coefficients();
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            const R c1 = C[coeff_at(q, 1)];
            pq[q] = pair2<R>(fma_(c1, cr.x, C[coeff_at(q, 0)]), c1);
        }
        cr.terms([&](int k, const v2<R> &td) {
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                const R c = C[coeff_at(q, k)];
                pq[q] = fma2(pair2<R>(c, c), td, pq[q]);
            }
        });
        h1 = cr.fch * pq[1].x; h2 = cr.fch * pq[2].x; h3 = cr.fch * pq[3].x; h4 = cr.fch * pq[4].x;
        dfch = cr.dfch;
        dxf = cr.dxf;
    } else {
        R f[NK], df[NK];
        carrier_fd2(r, P.inv_rc_r, f, df);
        load_coefficients();
#pragma unroll
        for (int q = 0; q < 4; ++q) he[q] = pair2<R>(R(0), R(0));
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            e0 += C[coeff_at(0, k)] * df[k];
            const v2<R> fd = pair2<R>(f[k], df[k]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const R c = C[coeff_at(q + 1, k)];
                he[q] = fma2(pair2<R>(c, c), fd, he[q]);
            }
        }
        h1 = he[0].x; h2 = he[1].x; h3 = he[2].x; h4 = he[3].x;
    }
    const R sij = si.x * sj.x + si.y * sj.y + si.z * sj.z;
    const R siu = si.x * ux + si.y * uy + si.z * uz;
    const R sju = sj.x * ux + sj.y * uy + sj.z * uz;
    const R wx = si.y * sj.z - si.z * sj.y, wy = si.z * sj.x - si.x * sj.z, wz = si.x * sj.y - si.y * sj.x;
    const R wu = wx * ux + wy * uy + wz * uz;
    R rad;
    if constexpr (sizeof(R) == 8) {
        const R phi[5] = {R(1), sij, wu, siu * sju, siu * siu};
#pragma unroll
        for (int q = 1; q < 5; ++q) pq[0] = fma2(pair2<R>(phi[q], phi[q]), pq[q], pq[0]);
        rad = fma_(dxf, pq[0].y, dfch * pq[0].x);
    } else {
        rad = e0 + he[0].y * sij + he[1].y * wu + he[2].y * siu * sju + he[3].y * siu * siu;
    }
    const R cSi = (h3 * sju + R(2) * h4 * siu) * ir;
    const R cSj = h3 * siu * ir;
    const R cW = h2 * ir;
    const R along = rad - cSi * siu - cSj * sju - cW * wu;
    R Dx = along * ux + cSi * si.x + cSj * sj.x + cW * wx;
    R Dy = along * uy + cSi * si.y + cSj * sj.y + cW * wy;
    R Dz = along * uz + cSi * si.z + cSj * sj.z + cW * wz;
    R cg = h1;   // coefficient of S_i in dE_i/dS_j (exchange, plus the spin-angular weight below)
    const R cu = h3 * sju + R(2) * h4 * siu;
    acc.hx += h1 * sj.x + h2 * (sj.y * uz - sj.z * uy) + cu * ux;
    acc.hy += h1 * sj.y + h2 * (sj.z * ux - sj.x * uz) + cu * uy;
    acc.hz += h1 * sj.z + h2 * (sj.x * uy - sj.y * ux) + cu * uz;
    if constexpr (ANG) {
        R g[NCH], dg[NCH];
        if (ti == 0) {
            if (tj == 0) ang_gdg<R, 0, 0>(P, r, P.inv_rc_a, g, dg);
            else ang_gdg<R, 0, 1>(P, r, P.inv_rc_a, g, dg);
        } else {
            if (tj == 0) ang_gdg<R, 1, 0>(P, r, P.inv_rc_a, g, dg);
            else ang_gdg<R, 1, 1>(P, r, P.inv_rc_a, g, dg);
        }
        R accu, avx, avy, avz, cj;
        if constexpr (sizeof(R) == 8) {
            bwd_angular<R>(sm, ux, uy, uz, sij, g, dg, accu, avx, avy, avz, cj);
        } else {
            v2<R> al = pair2<R>(R(0), R(0));
            avx = avy = avz = cj = R(0);
            v4<R> mid;
            bwd_harm<R, 0>(sm, ux, uy, uz, sij, g, dg, al, avx, avy, avz, cj, mid);
            accu = al.x + sij * al.y;
        }
        accu -= ir * (ux * avx + uy * avy + uz * avz);   // only the part across u turns the pair
        Dx += accu * ux + ir * avx;
        Dy += accu * uy + ir * avy;
        Dz += accu * uz + ir * avz;
        cg += cj;
        acc.hx += cj * sj.x;
        acc.hy += cj * sj.y;
        acc.hz += cj * sj.z;
    }
    // dE_i/dS_j = (h_EX + c_ij) S_i + h_DMI (u x S_i) + h_ANI (S_i.u) u
    const R Gx = cg * si.x + h2 * (uy * si.z - uz * si.y) + h3 * siu * ux;
    const R Gy = cg * si.y + h2 * (uz * si.x - ux * si.z) + h3 * siu * uy;
    const R Gz = cg * si.z + h2 * (ux * si.y - uy * si.x) + h3 * siu * uz;
    acc.fx += Dx; acc.fy += Dy; acc.fz += Dz;
    if constexpr (VIR) {
        acc.w[0] -= dx * Dx; acc.w[1] -= dx * Dy; acc.w[2] -= dx * Dz;
        acc.w[3] -= dy * Dx; acc.w[4] -= dy * Dy; acc.w[5] -= dy * Dz;
        acc.w[6] -= dz * Dx; acc.w[7] -= dz * Dy; acc.w[8] -= dz * Dz;
    }
    PairRec<R> *rec = a.pd + (int64_t)t * a.n + j;
    v4<R> ra, rb;
    ra.x = Dx; ra.y = Dy; ra.z = Dz; ra.w = Gx;
    rb.x = Gy; rb.y = Gz; rb.z = R(0); rb.w = R(0);
    store_rec(rec, ra, rb);
}

// rows lo, lo + LPA, ... of one range for one lane.  Two-level prefetch: the list entry of the
// row two steps ahead and the coordinates of the next row are in flight while a pair is
// computed, so no load waits on a load issued in the same step.
template <typename R, bool ANG, bool VIR, int LPA>
__device__ __forceinline__ void bwd_rows(const NepDev<R> &P, const Eval2Args<R> &a, int64_t i, int ti, int lo, int hi,
                                         int split, const v4<R> &pi, const v4<R> &si, const R *sm,
                                         BwdAcc2<R> &acc) {
    const int64_t N = a.n;
    const int2 *__restrict__ crow = a.crow + i;
    int2 e1 = make_int2(0, 0), e2 = e1, e3 = e1;   // (neighbour, the record's slot in its list)
    v4<R> p1, s1, p2, s2;
    if (lo < hi) e1 = ro(crow + (int64_t)lo * N);
    if (lo + LPA < hi) e2 = ro(crow + (int64_t)(lo + LPA) * N);
    if (lo + 2 * LPA < hi) e3 = ro(crow + (int64_t)(lo + 2 * LPA) * N);
    if (lo < hi) {
        pair_at(a, e1.x, p1, s1);
    }
    if (lo + LPA < hi) {
        pair_at(a, e2.x, p2, s2);
    }
#pragma unroll 1
    for (int row = lo; row < hi; row += LPA) {
        const int j = e1.x, t = e1.y;
        const v4<R> pj = p1, sj = s1;
        e1 = e2; p1 = p2; s1 = s2;
        e2 = e3;
        if (row + 2 * LPA < hi) {
            pair_at(a, e2.x, p2, s2);
        }
        if (row + 3 * LPA < hi) e3 = ro(crow + (int64_t)(row + 3 * LPA) * N);
        bwd_pair<R, ANG, VIR>(P, a, ti, row < split ? 0 : 1, pi, si, pj, sj, j, t, sm, acc);
    }
}

template <typename R, bool VIR, int LPA>
__device__ __forceinline__ void bwd_body(const NepDev<R> &P, const Eval2Args<R> &args, int64_t blk,
                                         unsigned char *smem_raw) {
    // the arguments as values: read once from the block's copy, so nothing in the loops below
    // depends on where they are stored
    const Eval2Args<R> a = args;
    if (a.skip && *a.skip) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int APW = 32 / LPA;   // atoms per warp
    const int grp = lane / LPA, ql = lane % LPA;
    const int64_t i = (blk * (blockDim.x >> 5) + warp) * APW + grp;
    const bool valid = i < a.n;
    const int64_t N = a.n;
    R *sm = reinterpret_cast<R *>(smem_raw) + warp * (LPA == 4 ? BW_WARP : BW_ATOM) + bwd_at<LPA>(grp);
    // the atom's lanes
    [[maybe_unused]] const unsigned quad = LPA == 32 ? 0xffffffffu : ((1u << (LPA & 31)) - 1u) << (grp * LPA);
    // FP32, four lanes per atom: both centres' coefficients in shared memory, after the atoms' (read
    // from global memory where they are used they came to 1.70 ms at 884,736 atoms)
    [[maybe_unused]] R *ctab = reinterpret_cast<R *>(smem_raw) + (blockDim.x >> 5) * BW_WARP;
    if constexpr (sizeof(R) == 4 && LPA == 4) {
        const v4<R> *src = reinterpret_cast<const v4<R> *>(a.ctab + CTAB_BWD);
        for (int e = threadIdx.x; e < NS * CB_CENTRE / 4; e += blockDim.x) reinterpret_cast<v4<R> *>(ctab)[e] = ro(src + e);
        __syncthreads();
    }
    BwdAcc2<R> acc;
    acc.fx = acc.fy = acc.fz = acc.hx = acc.hy = acc.hz = R(0);
#pragma unroll
    for (int t = 0; t < 9; ++t) acc.w[t] = R(0);
    if (valid) {
        const int ti = i < a.n_fe ? 0 : 1;
        v4<R> pi, si;
        pair_at(a, i, pi, si);
        const int4 c = ro(a.cnt + i);
        // the lane's gradient entries: of group R and of its own magnetic group (bwd_coeffs)
        const int qg = ql & 3;
        R fr[NCH], fm[NCH];
#pragma unroll
        for (int n = 0; n < NCH; ++n) {
            fr[n] = ro(a.fp + (int64_t)(Q_R + n) * N + i);
            fm[n] = ro(a.fp + (int64_t)(Q_EX + qg * NCH + n) * N + i);
        }
        // the angular channels' entries (dE/dq_A, dE/dq_SA)_n of degree l; four lanes per atom: lane
        // l - 1 fetches them for the others
        auto angular_entries = [&](int l, v4<R> &x0, v4<R> &x1, v2<R> &x2) {
            const R *fa = a.fp + (int64_t)(Q_A + l - 1) * N + i, *fs = a.fp + (int64_t)(Q_SA + l - 1) * N + i;
            x0.x = ro(fa); x0.y = ro(fs); x0.z = ro(fa + 4 * N); x0.w = ro(fs + 4 * N);
            x1.x = ro(fa + 8 * N); x1.y = ro(fs + 8 * N); x1.z = ro(fa + 12 * N); x1.w = ro(fs + 12 * N);
            x2.x = ro(fa + 16 * N); x2.y = ro(fs + 16 * N);
        };
        if constexpr (LPA == 4) {
            v4<R> x0, x1;
            v2<R> x2;
            angular_entries(ql + 1, x0, x1, x2);
            R *d = sm + BW_C + 12 * ql;
            reinterpret_cast<v4<R> *>(d)[0] = x0;
            reinterpret_cast<v4<R> *>(d)[1] = x1;
            *reinterpret_cast<v2<R> *>(d + 8) = x2;
            __syncwarp(quad);
        }
        // angular adjoints of this lane's harmonics (lm_of) from their records of ten entries: two neighbouring
        // harmonics' in five loads of four values, with a warp per atom one's in five of two
#pragma unroll
        for (int m = 0; m < (NLM + LPA - 1) / LPA; ++m) {
            const int lm = lm_of<LPA>(ql, m);
            if (LPA > 8 && lm >= NLM) break;
            const int64_t at = ((int64_t)i * NLM + lm) * BREC;
            v4<R> x0, x1;
            v2<R> x2;
            if constexpr (LPA == 4) {   // with its neighbour's record, in five pieces
                if (m % 2) continue;
                v4<R> w[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) w[q] = ro(reinterpret_cast<const v4<R> *>(a.bsum + at) + q);
                auto entries = [&](int l) {
                    const R *e = sm + BW_C + 12 * (l - 1);
                    x0 = reinterpret_cast<const v4<R> *>(e)[0];
                    x1 = reinterpret_cast<const v4<R> *>(e)[1];
                    x2 = *reinterpret_cast<const v2<R> *>(e + 8);
                };
                entries(l_of_lm(lm));
                const R k2 = R(2) * kappa_of_lm<R>(lm), k3 = R(2) * kappa_of_lm<R>(lm + 1);
                w[0].x *= k2 * x0.x; w[0].y *= k2 * x0.y; w[0].z *= k2 * x0.z; w[0].w *= k2 * x0.w;
                w[1].x *= k2 * x1.x; w[1].y *= k2 * x1.y; w[1].z *= k2 * x1.z; w[1].w *= k2 * x1.w;
                w[2].x *= k2 * x2.x; w[2].y *= k2 * x2.y;
                entries(l_of_lm(lm + 1));
                w[2].z *= k3 * x0.x; w[2].w *= k3 * x0.y;
                w[3].x *= k3 * x0.z; w[3].y *= k3 * x0.w; w[3].z *= k3 * x1.x; w[3].w *= k3 * x1.y;
                w[4].x *= k3 * x1.z; w[4].y *= k3 * x1.w; w[4].z *= k3 * x2.x; w[4].w *= k3 * x2.y;
                v4<R> *d = reinterpret_cast<v4<R> *>(sm + BREC * lm);
#pragma unroll
                for (int q = 0; q < 5; ++q) d[q] = w[q];
            } else {
                angular_entries(l_of_lm(lm), x0, x1, x2);
                const R k2 = R(2) * kappa_of_lm<R>(lm);
                const v2<R> e[NCH] = {pair2<R>(x0.x, x0.y), pair2<R>(x0.z, x0.w), pair2<R>(x1.x, x1.y),
                                      pair2<R>(x1.z, x1.w), x2};
#pragma unroll
                for (int n = 0; n < NCH; ++n) {
                    v2<R> w = ro(reinterpret_cast<const v2<R> *>(a.bsum + at) + n);
                    w.x *= k2 * e[n].x; w.y *= k2 * e[n].y;
                    reinterpret_cast<v2<R> *>(sm + BREC * lm)[n] = w;
                }
            }
        }
        if constexpr (LPA == 4) __syncwarp(quad);   // the entries are read: the coefficients take their place
        if (ql == 0) {   // onsite term dE_i/dS_i = 2 Fp_O S_i, counted once per atom
            const R fo = R(2) * ro(a.fp + (int64_t)Q_O * N + i);
            acc.hx = fo * si.x; acc.hy = fo * si.y; acc.hz = fo * si.z;
        }
        if constexpr (LPA == 4) {
            if constexpr (sizeof(R) == 4)
                bwd_coeffs<R, NS>(ctab + ti * CB_CENTRE, fm, fr, ql, 0, sm + BW_C);
            else
                bwd_coeffs<R, NS>(a.ctab + CTAB_BWD + ti * CB_CENTRE, fm, fr, ql, 0, sm + BW_C);
        } else if (ql < 4 * NS) {   // four lanes per neighbour species
            bwd_coeffs<R, 1>(a.ctab + CTAB_BWD + ti * CB_CENTRE, fm, fr, qg, ql >> 2, sm + BW_C);
        }
        __syncwarp(quad);
        const int ca = a.cap_ang;
        bwd_rows<R, true, VIR, LPA>(P, a, i, ti, ql, c.y, c.x, pi, si, sm, acc);
        bwd_rows<R, false, VIR, LPA>(P, a, i, ti, ca + ql, ca + c.w, ca + c.z, pi, si, sm, acc);
    }
    // per-atom sums over the atom's lanes
#pragma unroll
    for (int o = 1; o < LPA; o <<= 1) {
        acc.fx += __shfl_xor_sync(0xffffffffu, acc.fx, o);
        acc.fy += __shfl_xor_sync(0xffffffffu, acc.fy, o);
        acc.fz += __shfl_xor_sync(0xffffffffu, acc.fz, o);
        acc.hx += __shfl_xor_sync(0xffffffffu, acc.hx, o);
        acc.hy += __shfl_xor_sync(0xffffffffu, acc.hy, o);
        acc.hz += __shfl_xor_sync(0xffffffffu, acc.hz, o);
    }
    if constexpr (VIR) {
#pragma unroll
        for (int t = 0; t < 9; ++t)
#pragma unroll
            for (int o = 1; o < LPA; o <<= 1) acc.w[t] += __shfl_xor_sync(0xffffffffu, acc.w[t], o);
    }
    if (valid && ql == 0) {
        v4<R> f4, g4;
        f4.x = acc.fx; f4.y = acc.fy; f4.z = acc.fz; f4.w = R(0);
        g4.x = acc.hx; g4.y = acc.hy; g4.z = acc.hz; g4.w = R(0);
        stg(a.fown + i, f4);
        stg(a.gii + i, g4);
        if constexpr (VIR) {
#pragma unroll
            for (int t = 0; t < 9; ++t) stg(a.wpart + (int64_t)t * N + i, acc.w[t]);
        }
    }
}


// The evaluation kernels over an argument table (sl_batch.h: a system's own table or a
// batch's).  MINB: the register budget, as the minimum resident blocks per SM.  The
// mixed-precision kernels default to 4 blocks (128 registers) and have a second budget each,
// which sl_autotune may choose: radial (one thread per atom) and backward 3 blocks, angular
// unconstrained.
template <int MINB = 4>
__global__ void __launch_bounds__(128, MINB) k_crad(const __grid_constant__ NepDev<float> P,
                                                    const Eval2Args<float> *__restrict__ tab, SlotMap sm,
                                                    const __grid_constant__ Eval2Args<float> solo) {
    __shared__ uint32_t smask[MASKW_MAX][128];   // blocks have at most 128 threads
    one_work(tab, sm, solo, [&](const Eval2Args<float> &a, int64_t blk, int64_t) { crad_body(P, a, blk, smask); });
}
template <typename R>   // (blocks of these three have at most 128 threads)
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 8 : 4) k_crad_wide(const __grid_constant__ NepDev<R> P,
                                                                           const Eval2Args<R> *__restrict__ tab,
                                                                           SlotMap sm,
                                                                           const __grid_constant__ Eval2Args<R> solo) {
    __shared__ __align__(32) CradSmem<R> scratch;
    __shared__ CradRowsSmem rows;
    __shared__ CradLists lists;
    one_work(tab, sm, solo, [&](const Eval2Args<R> &a, int64_t blk, int64_t) { crad_wide_body(P, a, blk, scratch, rows, lists); });
}
template <typename R>
__global__ void __launch_bounds__(128, 8) k_crad_rows(const __grid_constant__ NepDev<R> P, const Eval2Args<R> *__restrict__ tab,
                                                      SlotMap sm, const __grid_constant__ Eval2Args<R> solo) {
    __shared__ CradRowsSmem rows;
    one_work(tab, sm, solo, [&](const Eval2Args<R> &a, int64_t blk, int64_t) { crad_rows_body(P, a, blk, rows); });
}
template <typename R>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 8 : 4) k_crad_sums(const __grid_constant__ NepDev<R> P,
                                                                           const Eval2Args<R> *__restrict__ tab,
                                                                           SlotMap sm,
                                                                           const __grid_constant__ Eval2Args<R> solo) {
    __shared__ __align__(32) CradSmem<R> scratch;
    one_work(tab, sm, solo, [&](const Eval2Args<R> &a, int64_t blk, int64_t) { crad_sums_body(P, a, blk, scratch); });
}
template <typename R, int MINB = sizeof(R) == 4 ? 4 : 1>
__global__ void __launch_bounds__(128, MINB) k_ang_fwd(const __grid_constant__ NepDev<R> P,
                                                       const Eval2Args<R> *__restrict__ tab, SlotMap sm,
                                                       const __grid_constant__ Eval2Args<R> solo) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    one_work(tab, sm, solo,
             [&](const Eval2Args<R> &a, int64_t blk, int64_t) { ang_fwd_body<R, 4>(P, a, blk, smem_raw); });
}
template <typename R, int MINB = sizeof(R) == 4 ? 4 : 1, bool VIR = false>
__global__ void __launch_bounds__(128, MINB) k_bwd(const __grid_constant__ NepDev<R> P,
                                                   const Eval2Args<R> *__restrict__ tab, SlotMap sm,
                                                   const __grid_constant__ Eval2Args<R> solo) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    one_work(tab, sm, solo,
             [&](const Eval2Args<R> &a, int64_t blk, int64_t) { bwd_body<R, VIR, 4>(P, a, blk, smem_raw); });
}

// The same with a warp per atom, for systems too small to fill the GPU four lanes per atom (the line
// in eval_is_wide).  FP64 at 512 / 1,728 / 2,744 atoms: angular 32 / 71 / 110 instead of 117 / 120 / 140
// us, backward 75 / 198 / 321 instead of 380 / 387 / 398 us (its 21 angular pairs fill two thirds of a
// round of 32 lanes, so in larger systems four lanes need fewer FP64 instructions).  Mixed precision
// at 512 / 1,728 / 2,744 / 4,096 atoms: angular 10 / 10 / 14.5 / 16 instead of 12 / 12 / 12 / 12 us,
// backward 12 / 15 / 20 / 27 instead of 23 / 24 / 24 / 25 us.  One line serves both kernels: in mixed precision, at
// 2,048 atoms, below where their sum crosses (2,744 atoms: 34.5 against 36 us); in FP64, at 3,040, little
// above the largest size timed, where both still gain.
template <typename R>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 4 : 1) k_ang_wide(const __grid_constant__ NepDev<R> P,
                                                                          const Eval2Args<R> *__restrict__ tab,
                                                                          SlotMap sm,
                                                                          const __grid_constant__ Eval2Args<R> solo) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    one_work(tab, sm, solo,
             [&](const Eval2Args<R> &a, int64_t blk, int64_t) { ang_fwd_body<R, 32>(P, a, blk, smem_raw); });
}
template <typename R, bool VIR = false>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 3 : 1) k_bwd_wide(const __grid_constant__ NepDev<R> P,
                                                                          const Eval2Args<R> *__restrict__ tab,
                                                                          SlotMap sm,
                                                                          const __grid_constant__ Eval2Args<R> solo) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    one_work(tab, sm, solo,
             [&](const Eval2Args<R> &a, int64_t blk, int64_t) { bwd_body<R, VIR, 32>(P, a, blk, smem_raw); });
}

// ------------------------------------------------------------------ launch
// The arguments of an evaluation at `at` (null members: the state).
template <typename R>
static Eval2Args<R> args2(Sys &s, const EvalAt &at, bool want_virial) {
    Eval2Args<R> a;
    if constexpr (sizeof(R) == 8) {
        a.pos = reinterpret_cast<const v4<R> *>(at.pos ? at.pos : s.pos);
        a.spin = reinterpret_cast<const v4<R> *>(at.spin ? at.spin : s.spin);
        a.box = *reinterpret_cast<const BoxDev<R> *>(&s.boxd);
        a.boxf = s.boxf;
    } else {
        a.pos = reinterpret_cast<const v4<R> *>(at.psf ? at.psf : s.psf);
        a.spin = a.pos + 1;
        a.box = *reinterpret_cast<const BoxDev<R> *>(&s.boxf);
    }
    a.posf = at.posf ? at.posf : s.posf;
    a.split = crad_is_split(s);
    a.skip = at.skip;
    a.nbr = s.nbr; a.seg = s.seg; a.rev = s.rev; a.capr = nbr_stride(s.cap); a.n = s.n; a.n_fe = s.n_fe;
    a.cap = s.cap; a.cap_ang = s.cap_ang;
    a.crow = s.crow; a.ctab = (const R *)s.ctab; a.cnt = s.cnt; a.mask = s.cmask; a.maskw = s.maskw;
    a.q = (R *)s.q; a.qs = s.qs; a.bsum = (R *)s.bsum; a.fp = (R *)s.fp; a.ei = (R *)s.ei;
    a.pd = (PairRec<R> *)s.pairs; a.fown = (v4<R> *)s.fown; a.gii = (v4<R> *)s.gii;
    a.wpart = (R *)s.wpart; a.want_virial = want_virial; a.status = s.status;
    return a;
}

template <typename R>
static constexpr int quad_block() { return sizeof(R) == 8 ? 64 : 128; }
template <typename R>
static constexpr size_t fwd_smem(int qb = quad_block<R>()) { return (size_t)(qb / 32) * FWARP * sizeof(R); }
template <typename R>
static constexpr size_t bwdf_smem(int qb = quad_block<R>()) {
    return ((size_t)(qb / 32) * BW_WARP + (sizeof(R) == 4 ? NS * CB_CENTRE : 0)) * sizeof(R);
}
template <typename R>
static constexpr size_t bwdw_smem(int qb) { return (size_t)(qb / 32) * BW_ATOM * sizeof(R); }

int default_quad_block(int prec) { return prec == 0 ? quad_block<double>() : quad_block<float>(); }

// Dynamic shared-memory limits of the quad kernels, set once per device (function
// attributes belong to the device's context), safe to call from several threads.
void eval2_init() {
    static std::mutex mu;
    static uint64_t done = 0;   // bit d: device d is set up
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 64 && (done >> dev & 1u)) return;
    cudaFuncSetAttribute(k_ang_fwd<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd_smem<float>());
    cudaFuncSetAttribute(k_ang_fwd<float, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd_smem<float>());
    cudaFuncSetAttribute(k_ang_fwd<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd_smem<double>());
    cudaFuncSetAttribute(k_bwd<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bwdf_smem<float>());
    cudaFuncSetAttribute(k_bwd<float, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bwdf_smem<float>());
    cudaFuncSetAttribute(k_bwd<float, 4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bwdf_smem<float>());
    cudaFuncSetAttribute(k_bwd<float, 3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bwdf_smem<float>());
    cudaFuncSetAttribute(k_bwd<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bwdf_smem<double>());
    cudaFuncSetAttribute(k_bwd<double, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)bwdf_smem<double>());
    cudaFuncSetAttribute(k_ang_wide<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd_smem<float>());
    cudaFuncSetAttribute(k_ang_wide<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd_smem<double>());
    if (dev < 64) done |= 1ull << dev;
}

// ---- argument tables (sl_batch.h)
size_t fused_eval_size(int prec) { return prec == 0 ? sizeof(Eval2Args<double>) : sizeof(Eval2Args<float>); }

// slot kinds: the step's evaluation (at the state, no virial), the full one (with the virial
// parts) and the midpoint iteration's (at its point, with its skip flag)
static EvalAt eval_point(const Sys &s, int kind) {
    EvalAt at;
    if (kind == SK_MID && s.mid_iters > 0) {
        at.pos = s.posmid; at.spin = s.mids; at.posf = s.midposf; at.psf = s.midpsf;
        at.skip = reinterpret_cast<const int *>(reinterpret_cast<const char *>(s.md) + offsetof(MidDev, converged));
    }
    return at;
}

void fused_put_eval(Sys &s, int r, int kind, const FusedTables &t, unsigned char *img, int64_t *blocks) {
    const EvalAt at = eval_point(s, kind);
    if (s.prec == 0) reinterpret_cast<Eval2Args<double> *>(img + t.o_eval)[r] = args2<double>(s, at, kind == SK_FULL);
    else reinterpret_cast<Eval2Args<float> *>(img + t.o_eval)[r] = args2<float>(s, at, kind == SK_FULL);
    const int qb = default_quad_block(s.prec);
    const bool wide = crad_is_wide(s);
    blocks[FK_CRAD] = wide ? 0 : (s.n + 127) / 128;
    blocks[FK_CRADW] = wide ? (s.n + CRAD_WIDE_ATOMS - 1) / CRAD_WIDE_ATOMS : 0;
    const bool warp = eval_is_wide(s);   // a warp per atom
    blocks[FK_ANG] = blocks[FK_BWD] = warp ? 0 : (s.n + qb / 4 - 1) / (qb / 4);
    blocks[FK_ANGW] = blocks[FK_BWDW] = warp ? (s.n + qb / 32 - 1) / (qb / 32) : 0;
}

// Radial, angular, network and backward (and, last, the three wide kernels) over a table, each launch in its own shape
// (L[k].block threads, 0: the default) and register budget (L[k].minb, 0: the default).
template <typename R>
void launch_eval_t(const FusedTables &t, const NepDev<R> &P, const Launch *L, cudaStream_t st, cudaEvent_t *ev,
                   const Fork &fork, const Fork &fork2) {
    // a system's own launch passes its argument block as a kernel parameter; a batch's reads
    // the table (the same for the four kernels of one launch group)
    const Eval2Args<R> *tab = L[0].solo ? nullptr : t.at<Eval2Args<R>>(t.o_eval);
    const Eval2Args<R> so = solo_args<Eval2Args<R>>(L[0]);
    const SlotMap s0 = L[0].slots(), s1 = L[1].slots(), s3 = L[3].slots();
    const int cb = L[0].block ? L[0].block : 128;
    const int qa = L[1].block ? L[1].block : quad_block<R>();
    const int qw = L[3].block ? L[3].block : quad_block<R>();
    if (ev) cudaEventRecord(ev[0], st);
    // compaction and radial channels in one kernel: the compaction group is empty
    if (ev) cudaEventRecord(ev[1], st);
    // a system's own launch has a grid for one kernel of each kind only; a batch's two, over different
    // slots, run side by side (the wider ones on the fork's stream)
    cudaStream_t side = fork.open(st);
    if constexpr (sizeof(R) == 4) {
        if (L[0].grid && L[0].minb == 3) k_crad<3><<<L[0].grid, cb, 0, st>>>(P, tab, s0, so);
        else if (L[0].grid) k_crad<<<L[0].grid, cb, 0, st>>>(P, tab, s0, so);
    }
    const int wb = L[4].block ? L[4].block : 128;
    // (a batch launches both forms: a slot's blocks return at once in the one it does not take)
    if (L[4].grid && !(L[4].solo && so.split)) k_crad_wide<R><<<L[4].grid, wb, 0, side>>>(P, tab, L[4].slots(), so);
    const bool split = L[4].grid && !(L[4].solo && !so.split);
    if (split) k_crad_rows<R><<<L[4].grid, wb, 0, side>>>(P, tab, L[4].slots(), so);
    fork.close(st);
    // the sums beside the angular kernels
    if (split) k_crad_sums<R><<<L[4].grid, wb, 0, side>>>(P, tab, L[4].slots(), so);
    bool variant = false;
    if (ev) cudaEventRecord(ev[2], st);
    const cudaStream_t side2 = fork2.open(st);
    if constexpr (sizeof(R) == 4) {
        variant = L[1].minb == 1 && L[1].grid;
        if (variant) k_ang_fwd<R, 1><<<L[1].grid, qa, fwd_smem<R>(qa), st>>>(P, tab, s1, so);
    }
    if (!variant && L[1].grid) k_ang_fwd<R><<<L[1].grid, qa, fwd_smem<R>(qa), st>>>(P, tab, s1, so);
    if (L[5].grid) {
        const int b = L[5].block ? L[5].block : quad_block<R>();
        k_ang_wide<R><<<L[5].grid, b, fwd_smem<R>(b), side2>>>(P, tab, L[5].slots(), so);
    }
    fork2.close(st);
    fork.close(st);
    if (ev) cudaEventRecord(ev[3], st);
    if constexpr (sizeof(R) == 4) launch_net_t_tc(t, P, L[2], st);
    else launch_net_t_fp64(t, L[2], st);
    if (ev) cudaEventRecord(ev[4], st);
    // the virial parts: only a system's own full evaluation asks for them (a batch's slots are
    // set up for the step's evaluation, which has none)
    const bool vir = L[3].solo && so.want_virial;
    side = fork.open(st);
    if (L[3].grid) {
        variant = false;
        if constexpr (sizeof(R) == 4) {
            variant = L[3].minb == 3;
            if (variant && vir) k_bwd<R, 3, true><<<L[3].grid, qw, bwdf_smem<R>(qw), st>>>(P, tab, s3, so);
            else if (variant) k_bwd<R, 3><<<L[3].grid, qw, bwdf_smem<R>(qw), st>>>(P, tab, s3, so);
        }
        if (!variant && vir)
            k_bwd<R, sizeof(R) == 4 ? 4 : 1, true><<<L[3].grid, qw, bwdf_smem<R>(qw), st>>>(P, tab, s3, so);
        else if (!variant) k_bwd<R><<<L[3].grid, qw, bwdf_smem<R>(qw), st>>>(P, tab, s3, so);
    }
    if (L[6].grid) {
        const int b = L[6].block ? L[6].block : quad_block<R>();
        if (vir) k_bwd_wide<R, true><<<L[6].grid, b, bwdw_smem<R>(b), side>>>(P, tab, L[6].slots(), so);
        else k_bwd_wide<R><<<L[6].grid, b, bwdw_smem<R>(b), side>>>(P, tab, L[6].slots(), so);
    }
    fork.close(st);
    if (ev) cudaEventRecord(ev[5], st);
}
template void launch_eval_t<float>(const FusedTables &, const NepDev<float> &, const Launch *, cudaStream_t,
                                   cudaEvent_t *, const Fork &, const Fork &);
template void launch_eval_t<double>(const FusedTables &, const NepDev<double> &, const Launch *, cudaStream_t,
                                    cudaEvent_t *, const Fork &, const Fork &);

// The system's own evaluation: at the midpoint point while s.at is set (the midpoint
// iteration), else at the state, with the virial parts when asked for.
void launch_eval(Sys &s, bool want_virial, cudaEvent_t *ev, bool forward_only) {
    if (s.n == 0) return;
    const int kind = s.at.pos ? SK_MID : want_virial ? SK_FULL : SK_STEP;
    Launch L[7] = {solo_launch(s, FK_CRAD, kind), solo_launch(s, FK_ANG, kind),   solo_launch(s, FK_NET, kind),
                   solo_launch(s, FK_BWD, kind),  solo_launch(s, FK_CRADW, kind), solo_launch(s, FK_ANGW, kind),
                   solo_launch(s, FK_BWDW, kind)};
    if (forward_only) L[3].grid = L[6].grid = 0;
    // (a profiled evaluation's kernels run one after the other)
    const Fork fork = crad_is_split(s) && !ev ? s.solo->fork : Fork();
    if (s.prec == 0) launch_eval_t<double>(s.solo->t, s.pd, L, s.stream, ev, fork);
    else launch_eval_t<float>(s.solo->t, s.pf, L, s.stream, ev, fork);
}

}  // namespace sl
