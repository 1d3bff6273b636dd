// sl_nep.cu -- the NEP-SPIN model, its CUDA-core network and the no-allocation evaluation.
//
// Descriptor of atom i (arXiv 2606.14073, Sections 5.1.1-5.1.2; 66 entries, Section 5.2.3):
//   R_n  = sum_j g^R_n(r_ij)                           radial, r < rc_rad
//   X_n  = sum_j g^X_n(r_ij) phi_X(S_i, S_j, u_ij)      X = EX, DMI, ANI, SIA (Section 5.2.4)
//   A_nl = sum_m kappa_lm B_nlm^2,   B_nlm  = sum_j g^A_n(r_ij) p_lm(u_ij)           r < rc_ang
//   SA_nl = sum_m kappa_lm BS_nlm^2, BS_nlm = sum_j g^A_n(r_ij) (S_i.S_j) p_lm(u_ij)
//   O = |S_i|^2
// with g^G_n = sum_k c^G_{n k t_i t_j} f_k (shared Chebyshev carrier, Section 5.2.4).
// The angular channels use the harmonic (addition-theorem) form: one pass over
// neighbours per channel n instead of the pair double sum.
//
// This file holds the no-allocation entry point's kernel (one warp per atom) and the
// CUDA-core network k_mlp:
//   E_i and Fp = dE_i/dq_i.
// The step's evaluation kernels are in sl_eval2.cu; forces and fields are gathered
// without atomics (sl_integrate.cu):
//   F_k = sum_j (dE_k/dr_kj - dE_j/dr_jk),  H_k = -dE_k/dS_k - sum_j dE_j/dS_k + Zeeman.
//
#include <cstddef>
#include <mutex>
#include <vector>

#include "sl_internal.h"
#include "sl_batch.h"
#include "sl_fused.cuh"

namespace sl {

// ------------------------------------------------------------------ network
// E_i = sum_h w1_h tanh(z_h) - b1, z_h = sum_v W0_hv s_v q_v - b0_h;
// Fp_v = s_v sum_h w1_h (1 - tanh^2 z_h) W0_hv.
// FP64 (the mixed-precision network runs on the tensor cores, sl_mlp_tc.cu): eight atoms per
// 128-thread block, two per warp.  The weights and the block's descriptors are staged in shared
// memory; lane h takes hidden unit h of both atoms, then the lanes take the 2 x 66 gradient
// entries, 32 at a time, and eight lanes share each of the last four.  What bounds it: the FP64
// pipe (160 warp instructions per atom; one thread per atom took 184, and a serial chain of 4,000
// multiply-adds however few the atoms): 512 / 13,824 / 110,592 atoms 25 / 154 / 984 us, against
// 202 / 228 / 1,070.
constexpr int NET_ATOMS = 8;          // atoms per block
constexpr int NET_LD = DIM + 1;       // row length of W0 in the table and in shared memory
// weight table of a system (device): W0 [NH][NET_LD], b0 [NH], w1 [NH], s [DIM], b1
constexpr int NT_B0 = NH * NET_LD, NT_W1 = NT_B0 + NH, NT_S = NT_W1 + NH, NT_B1 = NT_S + DIM, NT_SIZE = NT_B1 + 1;

template <typename R>
struct NetSmem {
    R w[NT_SIZE];
    R x[DIM][NET_ATOMS];       // s_v q_v, then the gradient entries
    R t[NET_ATOMS][NH];
};

template <typename R>
__device__ __forceinline__ void mlp_body(const NetArgs<R> &a, int64_t blk, NetSmem<R> &sm) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t i0 = blk * NET_ATOMS;
    for (int k = tid; k < NT_SIZE; k += 128) sm.w[k] = ro(a.wtab + k);
    for (int k = tid; k < DIM * NET_ATOMS; k += 128) {
        const int v = k / NET_ATOMS, c = k % NET_ATOMS;
        const R q = i0 + c < a.n ? a.q[(int64_t)v * a.qs + i0 + c] : R(0);
        sm.x[v][c] = q * ro(a.wtab + NT_S + v);
    }
    __syncthreads();
    const int c0 = 2 * warp, c1 = c0 + 1;   // the warp's atoms
    R E0 = R(0), E1 = R(0);
    if (lane < NH) {
        R z0 = -sm.w[NT_B0 + lane], z1 = z0;
        const R *w = sm.w + lane * NET_LD;
#pragma unroll 11
        for (int v = 0; v < DIM; ++v) {
            z0 += w[v] * sm.x[v][c0];
            z1 += w[v] * sm.x[v][c1];
        }
        const R t0 = tanh(z0), t1 = tanh(z1), w1 = sm.w[NT_W1 + lane];
        E0 = w1 * t0;
        E1 = w1 * t1;
        sm.t[c0][lane] = w1 * (R(1) - t0 * t0);
        sm.t[c1][lane] = w1 * (R(1) - t1 * t1);
    }
    // both atoms' sums over the units: the lower half of the warp takes the first atom's
    R E = (lane < 16 ? E0 : E1) + __shfl_xor_sync(0xffffffffu, lane < 16 ? E1 : E0, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) E += __shfl_xor_sync(0xffffffffu, E, o);
    const int64_t ie = i0 + c0 + (lane >> 4);
    if ((lane & 15) == 0 && ie < a.n) a.ei[ie] = E - sm.w[NT_B1];
    __syncwarp();   // this warp's descriptors are read, its t's written
#pragma unroll
    for (int r = 0; r < 4; ++r) {   // 2 x 64 gradient entries
        const int v = (r & 1) * 32 + lane, c = c0 + (r >> 1);
        R s = R(0);
#pragma unroll 10
        for (int h = 0; h < NH; ++h) s += sm.t[c][h] * sm.w[h * NET_LD + v];
        sm.x[v][c] = s * sm.w[NT_S + v];
    }
    {   // the last 2 x 2: eight lanes each
        const int v = 64 + (lane >> 3 & 1), c = c0 + (lane >> 4);
        R s = R(0);
        for (int h = lane & 7; h < NH; h += 8) s += sm.t[c][h] * sm.w[h * NET_LD + v];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((lane & 7) == 0) sm.x[v][c] = s * sm.w[NT_S + v];
    }
    __syncthreads();
    for (int k = tid; k < DIM * NET_ATOMS; k += 128) {
        const int v = k / NET_ATOMS, c = k % NET_ATOMS;
        if (i0 + c < a.n) a.fp[(int64_t)v * a.n + i0 + c] = sm.x[v][c];
    }
}

// over an argument table (sl_batch.h)
template <typename R>
__global__ void __launch_bounds__(128) k_mlp(const NetArgs<R> *__restrict__ tab, SlotMap sm,
                                             const __grid_constant__ NetArgs<R> solo) {
    __shared__ NetSmem<R> scratch;
    one_work(tab, sm, solo, [&](const NetArgs<R> &args, int64_t blk, int64_t) {
        const NetArgs<R> a = args;
        if (a.skip && *a.skip) return;
        mlp_body(a, blk, scratch);
    });
}

// the FP64 network's weight table, from the system's model; 0 on success
int make_net_table(Sys &s) {
    if (s.prec != 0 || s.n == 0) return 0;
    std::vector<double> t(NT_SIZE, 0.0);
    for (int h = 0; h < NH; ++h) {
        for (int v = 0; v < DIM; ++v) t[h * NET_LD + v] = s.pd.w0[h][v];
        t[NT_B0 + h] = s.pd.b0[h];
        t[NT_W1 + h] = s.pd.w1[h];
    }
    for (int v = 0; v < DIM; ++v) t[NT_S + v] = s.pd.scal[v];
    t[NT_B1] = s.pd.b1;
    if (!s.mlp_img && cudaMalloc(&s.mlp_img, sizeof(double) * NT_SIZE) != cudaSuccess) {
        s.mlp_img = nullptr;
        return -1;
    }
    if (cudaMemcpyAsync(s.mlp_img, t.data(), sizeof(double) * NT_SIZE, cudaMemcpyHostToDevice, s.stream) != cudaSuccess)
        return -1;
    return cudaStreamSynchronize(s.stream) == cudaSuccess ? 0 : -1;
}

// ---- argument tables (sl_batch.h): the FP64 network over NetArgs, the mixed one
// (sl_mlp_tc.cu) over MlpArgs holding each slot's TMA map
size_t fused_net_size(int prec) { return prec == 0 ? sizeof(NetArgs<double>) : sizeof(MlpArgs); }

void fused_put_net(Sys &s, int r, int kind, const FusedTables &t, unsigned char *img, int64_t *blocks) {
    // the midpoint iteration's evaluations stop once it has converged
    const int *skip = kind == SK_MID && s.md ? reinterpret_cast<const int *>(reinterpret_cast<const char *>(s.md) +
                                                                             offsetof(MidDev, converged))
                                             : nullptr;
    if (s.prec == 0) {
        NetArgs<double> a;
        a.q = (const double *)s.q; a.fp = (double *)s.fp; a.ei = (double *)s.ei; a.n = s.n; a.qs = s.qs;
        a.skip = skip; a.wtab = (const double *)s.mlp_img;
        reinterpret_cast<NetArgs<double> *>(img + t.o_net)[r] = a;
    } else {
        MlpArgs a;
        a.qmap = s.qmap; a.n = s.n; a.fp = (float *)s.fp; a.ei = (float *)s.ei; a.status = s.status;
        a.skip = skip; a.wimg = s.mlp_img;
        reinterpret_cast<MlpArgs *>(img + t.o_net)[r] = a;
    }
    const int per = s.prec == 0 ? NET_ATOMS : 128;   // atoms of a block, or of a tensor-core tile
    blocks[FK_NET] = (s.n + per - 1) / per;
}

static_assert(NET_ATOMS == CRAD_WIDE_ATOMS, "one atoms-per-block class in a batch (sl_batch.cu)");
void launch_net_t_fp64(const FusedTables &t, const Launch &L, cudaStream_t st) {
    k_mlp<double><<<L.grid, 128, 0, st>>>(L.solo ? nullptr : t.at<NetArgs<double>>(t.o_net), L.slots(),
                                          solo_args<NetArgs<double>>(L));
}

// ------------------------------------------------------------------ no-allocation variant
// Descriptors and network energies of a small system in ONE kernel that needs no device
// memory but a status word (a fixed file-scope device variable) beside its shared memory.  For
// callers that may not allocate (see sl_descriptors_energies_noalloc in spinlat.h).  Computes
// in FP64.
//
// One warp per atom, four atoms per block.  What bounds it: the FP64 pipe (two lanes per SM
// and cycle, so a warp's FP64 instruction takes 16 cycles of its SM); every stage therefore
// keeps as many of the 32 lanes busy as it can, and what is not FP64 arithmetic of the result
// stays off that pipe:
//   search    all pairs, FP32 separations of the staged positions; only pairs within the
//             rounding band around the cutoff take the exact FP64 test;
//   pairs     lanes over pairs, 32 at a time: geometry, carrier and spin products, staged in
//             shared memory;
//   sums      lanes over (k, third of the staged pairs): five group sums each; in the angular
//             part over (channel, four harmonics): eight sums each;
//   network   lanes over hidden units.
// A call on 1,000 atoms takes 0.13 ms, host side included; with one thread per atom (16 blocks
// at most, the search and the angular channels serial in each thread) it took 6.2 ms.
namespace noalloc {

constexpr int MAX_ATOMS = 2048;
constexpr int MAX_NBR = 160;   // neighbours inside rc_rad per atom
constexpr int WARPS = 4;       // atoms (warps) per block
constexpr int LD = 33;         // row length of a staged entry: 32 pairs and a pad against bank conflicts
constexpr int STAGE = 34 * LD; // angular stage: g_n, s g_n, the 24 harmonics (the radial one has 13 rows)
constexpr int W0_LD = DIM + 1;
constexpr int NCOEF = NS * NS * 6 * NCH * NK;

// The status word of a call, held by every GPU that loads the library until the process exits.
static __device__ int g_status;

struct WarpSmem {
    double stage[STAGE];
    double sums[NS][5][NK];      // radial and pairwise-magnetic basis sums per neighbour species
    double q[DIM];
    uint16_t list[MAX_NBR];      // neighbours inside rc_rad: species 0 from the front, species 1 from the back
    uint16_t ang[MAX_NBR];       // those inside rc_ang (positions in the walk over the list)
};
struct BlockSmem {
    double c[NCOEF];             // coefficients, as in NepDev
    double w0[NH * W0_LD];
    WarpSmem w[WARPS];
    float far[WARPS];
};

__device__ __forceinline__ double kappa_of(int lm) {
    switch (lm) {   // kappa_lm of the addition theorem
    case 0: case 1: case 2: return 1.0;
    case 3: case 4: case 5: return 3.0;
    case 6: return 0.75;
    case 8: case 14: case 18: case 20: return 0.625;
    case 9: return 15.0;
    case 10: case 12: return 0.375;
    case 7: case 11: return 0.25;
    case 13: return 3.75;
    case 15: return 8.75;
    case 16: case 22: return 4.375;
    case 17: return 1.25;
    case 19: return 0.015625;
    case 21: return 0.3125;
    default: return 0.546875;
    }
}

__global__ void __launch_bounds__(WARPS * 32) k_eval_noalloc(const __grid_constant__ NepDev<double> P,
                                                             const double4 *__restrict__ pos,
                                                             const double4 *__restrict__ spin,
                                                             const int32_t *__restrict__ species, int n,
                                                             BoxDev<double> box, int *status,
                                                             double *__restrict__ q_out,
                                                             double *__restrict__ e_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BlockSmem &sm = *reinterpret_cast<BlockSmem *>(smem_raw);
    float4 *fpos = reinterpret_cast<float4 *>(smem_raw + (sizeof(BlockSmem) + 15) / 16 * 16);   // [n]
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    WarpSmem &ws = sm.w[w];

    // FP32 positions of every atom, along periodic axes first brought into [-L/2, L/2] in FP64,
    // species in w; `far`: the largest coordinate, which sets the band of the FP32 test
    float far = 0.f;
    for (int j = tid; j < n; j += WARPS * 32) {
        const double4 p = pos[j];
        // (the whole box lengths in FP32: one off, should they be, only widens the band)
        const float px = (float)p.x, py = (float)p.y, pz = (float)p.z;
        const float x = (float)fma(-box.L[0], (double)rintf(px * (float)box.invL[0]), p.x),
                    y = (float)fma(-box.L[1], (double)rintf(py * (float)box.invL[1]), p.y),
                    z = (float)fma(-box.L[2], (double)rintf(pz * (float)box.invL[2]), p.z);
        const int t = species[j];
        // a species outside the model is reported and the host rejects the whole call
        if (t < 0 || t >= NS) atomicOr(status, ST_BAD_SPECIES);
        fpos[j] = make_float4(x, y, z, __int_as_float(t & 1));
        far = fmaxf(far, fmaxf(fmaxf(fabsf(x), fabsf(y)), fabsf(z)));
        // the exact test's own rounding, should a caller's coordinates span many boxes
        far = fmaxf(far, 1e-8f * fmaxf(fmaxf(fabsf(px), fabsf(py)), fabsf(pz)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) far = fmaxf(far, __shfl_xor_sync(0xffffffffu, far, o));
    if (lane == 0) sm.far[w] = far;
    const double *cin = &P.c[0][0][0][0][0];
    for (int k = tid; k < NCOEF; k += WARPS * 32) sm.c[k] = cin[k];
    for (int k = tid; k < NH * DIM; k += WARPS * 32) sm.w0[k / DIM * W0_LD + k % DIM] = P.w0[k / DIM][k % DIM];
    __syncthreads();
    const int i = blockIdx.x * WARPS + w;
    if (i >= n) return;   // no block-wide barrier below

    // ---- search.  An FP32 coordinate is off by 2^-24 of itself, a separation by the two
    // coordinates' errors, its own rounding (of at most twice the largest coordinate) and the
    // minimum image's (of a box length): at most E per component, so d2 (up to R^2, R a little
    // beyond the cutoff) by 2 sqrt(3) R E + 3 E^2 and the FP32 sum's 4 2^-24 R^2.  The band is
    // twice that.  A NaN fails both comparisons and takes the exact test.
    float lo, hi;
    {
        float m = 0.f, L = 0.f;
#pragma unroll
        for (int k = 0; k < WARPS; ++k) m = fmaxf(m, sm.far[k]);
#pragma unroll
        for (int a = 0; a < 3; ++a) L = fmaxf(L, box.invL[a] != 0.0 ? (float)box.L[a] : 0.f);
        const float u = 5.9604645e-8f, E = u * (4.f * m + 4.f * L), R = (float)P.rc_r + 1.f;
        const float band = 2.f * (3.4641017f * R * E + 3.f * E * E + 4.f * u * R * R);
        lo = (float)P.rc_r2 - band;
        hi = (float)P.rc_r2 + band;
    }
    const double4 pi = pos[i], si = spin[i];
    const float4 fi = fpos[i];
    const int ti = __float_as_int(fi.w);
    const BoxDev<float> bf = {{(float)box.L[0], (float)box.L[1], (float)box.L[2]},
                              {(float)box.invL[0], (float)box.invL[1], (float)box.invL[2]}};
    auto separation = [&](const double4 &pj, double &dx, double &dy, double &dz) {
        dx = pj.x - pi.x; dy = pj.y - pi.y; dz = pj.z - pi.z;
        minimg(box, dx, dy, dz);
        return dx * dx + dy * dy + dz * dz;
    };
    const unsigned lt = (1u << lane) - 1u;
    int m0 = 0, m1 = 0;
    for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        bool in = false, near = false;
        int tj = 0;
        if (j < n && j != i) {
            const float4 fj = fpos[j];
            float dx = fj.x - fi.x, dy = fj.y - fi.y, dz = fj.z - fi.z;
            minimg(bf, dx, dy, dz);
            const float d2 = dx * dx + dy * dy + dz * dz;
            in = d2 < lo;
            near = !in && !(d2 >= hi);
            tj = __float_as_int(fj.w);
        }
        if (near) {
            double dx, dy, dz;
            in = separation(pos[j], dx, dy, dz) < P.rc_r2;
        }
        const unsigned b0 = __ballot_sync(0xffffffffu, in && tj == 0), b1 = __ballot_sync(0xffffffffu, in && tj == 1);
        if (in) {
            const int at = tj == 0 ? m0 + __popc(b0 & lt) : m1 + __popc(b1 & lt);
            if (at < MAX_NBR) ws.list[tj == 0 ? at : MAX_NBR - 1 - at] = (uint16_t)j;
        }
        m0 += __popc(b0);
        m1 += __popc(b1);
    }
    if (m0 + m1 > MAX_NBR) {   // uniform over the warp; the host rejects the call
        if (lane == 0) atomicOr(status, ST_NBR_OVERFLOW);
        return;
    }
    const int m = m0 + m1;
    __syncwarp();
    auto neighbour = [&](int p) { return (int)ws.list[p < m0 ? p : MAX_NBR - 1 - (p - m0)]; };

    // ---- radial and pairwise-magnetic sums: 32 pairs staged at a time (f_k, then the four
    // spin products), summed by 27 lanes: lane (k, third) takes every third pair
    double s0[5] = {0, 0, 0, 0, 0}, s1[5] = {0, 0, 0, 0, 0};
    const int k9 = lane % 9, third = lane / 9;
    int na = 0;
    for (int base = 0; base < m; base += 32) {
        const int p = base + lane, cnt = min(32, m - base);
        bool ang = false;
        if (p < m) {
            const int j = neighbour(p);
            const double4 sj = spin[j];
            double dx, dy, dz;
            const double d2 = separation(pos[j], dx, dy, dz);
            ang = d2 < P.rc_a2;
            const double ir = rsqrt(d2), r = d2 * ir;
            const double ux = dx * ir, uy = dy * ir, uz = dz * ir;
            double f[NK];
            carrier_f(r, P.inv_rc_r, f);
#pragma unroll
            for (int k = 0; k < NK; ++k) ws.stage[k * LD + lane] = f[k];
            const double siu = si.x * ux + si.y * uy + si.z * uz, sju = sj.x * ux + sj.y * uy + sj.z * uz;
            ws.stage[9 * LD + lane] = si.x * sj.x + si.y * sj.y + si.z * sj.z;
            ws.stage[10 * LD + lane] = (si.y * sj.z - si.z * sj.y) * ux + (si.z * sj.x - si.x * sj.z) * uy +
                                       (si.x * sj.y - si.y * sj.x) * uz;
            ws.stage[11 * LD + lane] = siu * sju;
            ws.stage[12 * LD + lane] = siu * siu;
        }
        const unsigned ba = __ballot_sync(0xffffffffu, ang);
        if (ang) ws.ang[na + __popc(ba & lt)] = (uint16_t)p;
        na += __popc(ba);
        __syncwarp();
        if (third < 3) {
            const int split = min(max(m0 - base, 0), cnt);   // staged pairs of species 0
            auto add = [&](double *s, int at) {
                const double f = ws.stage[k9 * LD + at];
                s[0] += f;
#pragma unroll
                for (int g = 0; g < 4; ++g) s[g + 1] = fma(f, ws.stage[(9 + g) * LD + at], s[g + 1]);
            };
            for (int at = third; at < split; at += 3) add(s0, at);
            for (int at = split + third; at < cnt; at += 3) add(s1, at);
        }
        __syncwarp();
    }
#pragma unroll
    for (int g = 0; g < 5; ++g) {
        s0[g] += __shfl_sync(0xffffffffu, s0[g], (lane + 9) & 31) + __shfl_sync(0xffffffffu, s0[g], (lane + 18) & 31);
        s1[g] += __shfl_sync(0xffffffffu, s1[g], (lane + 9) & 31) + __shfl_sync(0xffffffffu, s1[g], (lane + 18) & 31);
        if (lane < 9) {
            ws.sums[0][g][lane] = s0[g];
            ws.sums[1][g][lane] = s1[g];
        }
    }
    __syncwarp();
    const double *ci = sm.c + ti * (NS * 6 * NCH * NK);   // [neighbour][group][n][k]
    if (lane < 25) {
        const int g = lane / NCH, c = lane % NCH;
        const int grp = g == 0 ? G_R : g + 1;                      // R, EX, DMI, ANI, SIA
        const int at = g == 0 ? Q_R : Q_EX + (g - 1) * NCH;
        double v = 0.0;
#pragma unroll
        for (int tj = 0; tj < NS; ++tj)
#pragma unroll
            for (int k = 0; k < NK; ++k) v += ci[((tj * 6 + grp) * NCH + c) * NK + k] * ws.sums[tj][g][k];
        ws.q[at + c] = v;
    }
    if (lane == 25) ws.q[Q_O] = si.x * si.x + si.y * si.y + si.z * si.z;

    // ---- angular sums: 32 pairs staged at a time (g_n, s g_n, harmonics), summed by 30 lanes:
    // lane (n, four harmonics)
    double B[4] = {0, 0, 0, 0}, BS[4] = {0, 0, 0, 0};
    const int nc = lane / 6, quad = lane % 6;
    for (int base = 0; base < na; base += 32) {
        const int cnt = min(32, na - base);
        if (lane < cnt) {
            const int p = ws.ang[base + lane], j = neighbour(p), tj = p < m0 ? 0 : 1;
            const double4 sj = spin[j];
            double dx, dy, dz;
            const double d2 = separation(pos[j], dx, dy, dz);
            const double ir = rsqrt(d2), r = d2 * ir;
            double f[NK];
            carrier_f(r, P.inv_rc_a, f);
            const double s = si.x * sj.x + si.y * sj.y + si.z * sj.z;
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
                double g = 0.0;
#pragma unroll
                for (int k = 0; k < NK; ++k) g += ci[((tj * 6 + G_A) * NCH + c) * NK + k] * f[k];
                ws.stage[c * LD + lane] = g;
                ws.stage[(NCH + c) * LD + lane] = g * s;
            }
            double h[NLM];
            harm_p(dx * ir, dy * ir, dz * ir, h);
#pragma unroll
            for (int lm = 0; lm < NLM; ++lm) ws.stage[(2 * NCH + lm) * LD + lane] = h[lm];
        }
        __syncwarp();
        if (nc < NCH) {
            for (int at = 0; at < cnt; ++at) {
                const double g = ws.stage[nc * LD + at], gs = ws.stage[(NCH + nc) * LD + at];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const double h = ws.stage[(2 * NCH + 4 * quad + x) * LD + at];
                    B[x] = fma(g, h, B[x]);
                    BS[x] = fma(gs, h, BS[x]);
                }
            }
        }
        __syncwarp();
    }
    if (nc < NCH) {   // the sums take the stage's place: B_n,lm, then BS_n,lm
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            ws.stage[nc * NLM + 4 * quad + x] = B[x];
            ws.stage[(NCH + nc) * NLM + 4 * quad + x] = BS[x];
        }
    }
    __syncwarp();
    for (int o = lane; o < 2 * NCH * 4; o += 32) {
        const int l = o & 3, c = o >> 2;   // c: channel n of A, then of SA
        const int lm0 = l * (l + 2), lm1 = (l + 1) * (l + 3);   // 0, 3, 8, 15, 24
        double v = 0.0;
        for (int lm = lm0; lm < lm1; ++lm) {
            const double b = ws.stage[c * NLM + lm];
            v += kappa_of(lm) * b * b;
        }
        ws.q[(c < NCH ? Q_A + c * 4 : Q_SA + (c - NCH) * 4) + l] = v;
    }
    __syncwarp();

    // ---- outputs and the network, E_i = sum_h w1_h tanh(sum_v W0_hv s_v q_v - b0_h) - b1
    for (int v = lane; v < DIM; v += 32) {
        const double x = ws.q[v];
        if (q_out) q_out[(int64_t)i * DIM + v] = x;
        ws.q[v] = x * P.scal[v];
    }
    __syncwarp();
    double E = 0.0;
    if (lane < NH) {
        double z0 = -P.b0[lane], z1 = 0.0;
#pragma unroll 6
        for (int v = 0; v < DIM; v += 2) {
            z0 = fma(sm.w0[lane * W0_LD + v], ws.q[v], z0);
            z1 = fma(sm.w0[lane * W0_LD + v + 1], ws.q[v + 1], z1);
        }
        E = P.w1[lane] * tanh(z0 + z1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) E += __shfl_xor_sync(0xffffffffu, E, o);
    if (lane == 0) e_out[i] = E - P.b1;
}

constexpr size_t smem_bytes(int n) { return (sizeof(BlockSmem) + 15) / 16 * 16 + sizeof(float4) * (size_t)n; }
static_assert(2 * smem_bytes(MAX_ATOMS) <= 227 * 1024, "two blocks share an SM at the largest size");

}  // namespace noalloc

// Device address of the status word for the current device, looked up once per device (host
// code cannot use the symbol itself as a device address), with the kernel's shared-memory limit.
static int noalloc_status(int **out) {
    static std::mutex mu;
    static void *addr[128] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) return -1;
    std::lock_guard<std::mutex> lk(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, noalloc::g_status) != cudaSuccess || !p) return -1;
        if (cudaFuncSetAttribute(noalloc::k_eval_noalloc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)noalloc::smem_bytes(noalloc::MAX_ATOMS)) != cudaSuccess)
            return -1;
        addr[dev] = p;
    }
    *out = static_cast<int *>(addr[dev]);
    return 0;
}

int launch_noalloc(const NepDev<double> &P, const double4 *pos, const double4 *spin, const int32_t *species, int n,
                   const BoxDev<double> &box, double *q_out, double *e_out, cudaStream_t stream, int *status_out) {
    int *status = nullptr;
    if (noalloc_status(&status)) return -1;
    if (cudaMemsetAsync(status, 0, sizeof(int), stream) != cudaSuccess) return -1;
    noalloc::k_eval_noalloc<<<(unsigned)((n + noalloc::WARPS - 1) / noalloc::WARPS), noalloc::WARPS * 32,
                              noalloc::smem_bytes(n), stream>>>(P, pos, spin, species, n, box, status, q_out, e_out);
    if (cudaGetLastError() != cudaSuccess) return -1;
    int st = 0;
    if (cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, stream) != cudaSuccess) return -1;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return -1;
    *status_out = st;
    return 0;
}

int noalloc_max_atoms() { return noalloc::MAX_ATOMS; }

}  // namespace sl
