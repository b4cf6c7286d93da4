// Analytic N-body sums of the energy partition (Sec. 3.3) and of the
// Coulomb / Debye-Hueckel boundary condition (Sec. 2.3).
//
//   Phi_t = sum_i q_i exp(-k r_ti) / r_ti          (k = 0: Coulomb)
//   Psi_t = sum_i q_i (r_t - r_i).n_t / r_ti^3      (dipole kernel, n_t = +-e_d,
//                                                    or the analytic surface normal)
//
// FP32 tiled kernel: sources staged in shared memory 256 at a time; each
// position is stored as an FP32 pair (hi + lo) relative to the grid centre so
// the difference r_t - r_i keeps ~46 bits; 1/r from rsqrtf; a tile's
// contributions are summed in groups of 16 in plain FP32, the group sums with
// Kahan compensation in FP32, and the tile sum is added to an FP64
// accumulator.  A thread's two targets share each
// instruction through the packed FP32x2 arithmetic of sm_100-class GPUs.
// It serves the surface terms Phi_p, Psi_p at the crossing points; of large
// sums it takes the near atoms only (nbody_far.cuh).
//
// FP64 kernels: the boundary values (they enter the linear system) and the
// Coulomb energy sum_{i<j} q_i q_j / r_ij (a net value of large terms of
// either sign), each summed in a fixed order.
#include <cub/block/block_reduce.cuh>
#include <cub/device/device_radix_sort.cuh>

#include <algorithm>

#include "fp64_math.cuh"
#include "pb_internal.h"

namespace pbg {

namespace {

constexpr int NB_THREADS = 256;
constexpr int NB_TPT = 2;  // targets per thread
constexpr int NB_GRP = 16; // sources per plainly summed group
// largest coordinate offset (A) of a block's targets from its first target
// for the per-block origin form of the differences
constexpr double NB_ORIGIN_EXT = 8.0;
// Octrees with at least so many pairs take local expansions for far atoms.
// Sorting the targets and the balls take about 0.2 ms: pairs and expansions both
// take 0.3 ms with 1,000 atoms (3.2e8 pairs), and 0.9 and 0.53 ms with 2,000 (1.2e9).
// Uniform grids keep all pairs: expansions there (0.52 instead of 0.99 ms at
// 257^3 with 2,000 atoms) were tried in a form whose near pairs had a larger
// error (Psi 1.57e-7 -> 1.89e-7 from 64 bits), and not since.
constexpr long long FAR_PAIRS = 400000000;

struct SrcHi {
    float x, y, z, q;
};
struct SrcLo {
    float x, y, z, pad;
};

__global__ void k_split_atoms(const double *__restrict__ atoms, long long na, double cx, double cy,
                              double cz, float4 *__restrict__ hi, float4 *__restrict__ lo) {
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= na) return;
    double c[3] = {atoms[i] - cx, atoms[na + i] - cy, atoms[2 * na + i] - cz};
    float h[3], l[3];
    for (int d = 0; d < 3; ++d) {
        h[d] = (float)c[d];
        l[d] = (float)(c[d] - (double)h[d]);
    }
    hi[i] = make_float4(h[0], h[1], h[2], (float)atoms[4 * na + i]);
    lo[i] = make_float4(l[0], l[1], l[2], 0.f);
}

// Target kinds
enum { TK_BOUNDARY = 0, TK_SURFACE = 1 };

struct TargetDesc {
    int kind;
    GridGeo g;
    double shift[3];
    // surface
    const double *rp;
    const long long *ids;
    const int8_t *sign;
    const double *nrm2; // optional second normal per target (PSI2): 3 per target
    const int *order;   // optional: the targets in the order in which blocks take them
    long long count;
};

__device__ __forceinline__ void boundary_node(const GridGeo &g, long long b, long long &i,
                                              long long &j, long long &k) {
    long long nxy = (long long)g.nx * g.ny;
    if (b < nxy) {
        i = b % g.nx;
        j = b / g.nx;
        k = 0;
        return;
    }
    if (b < 2 * nxy) {
        b -= nxy;
        i = b % g.nx;
        j = b / g.nx;
        k = g.nz - 1;
        return;
    }
    b -= 2 * nxy;
    long long ring = 2ll * g.nx + 2ll * (g.ny - 2);
    k = 1 + b / ring;
    long long q = b % ring;
    if (q < g.nx) {
        i = q;
        j = 0;
    } else if (q < 2ll * g.nx) {
        i = q - g.nx;
        j = g.ny - 1;
    } else {
        long long q2 = q - 2ll * g.nx;
        if (q2 < g.ny - 2) {
            i = 0;
            j = 1 + q2;
        } else {
            i = g.nx - 1;
            j = 1 + q2 - (g.ny - 2);
        }
    }
}

// the target at place t of the blocks' order (T.count: none)
__device__ __forceinline__ long long target_at(const TargetDesc &T, long long t) {
    return T.order && t < T.count ? T.order[t] : t;
}

struct TgtLoad {
    float h[3], l[3];
    float n[3];     // unit normal for Psi (surface targets)
    float n2[3];    // second normal (the analytic surface normal) when given
    bool active;    // contributes (flux edge / valid index)
};

__device__ __forceinline__ TgtLoad load_target(const TargetDesc &T, long long t) {
    TgtLoad r;
    double p[3] = {0.0, 0.0, 0.0};
    r.active = t < T.count;
    r.n[0] = r.n[1] = r.n[2] = 0.f;
    r.n2[0] = r.n2[1] = r.n2[2] = 0.f;
    if (r.active) {
        if (T.kind == TK_BOUNDARY) {
            long long i, j, k;
            boundary_node(T.g, t, i, j, k);
            p[0] = T.g.o[0] + (double)i * T.g.h;
            p[1] = T.g.o[1] + (double)j * T.g.h;
            p[2] = T.g.o[2] + (double)k * T.g.h;
        } else {
            int sg = T.sign[t];
            if (sg == 0) r.active = false;
            int d = (int)(T.ids[t] / T.g.N);
            r.n[d] = (float)sg;
            if (T.nrm2)
                for (int d = 0; d < 3; ++d) r.n2[d] = (float)T.nrm2[3 * t + d];
            p[0] = T.rp[3 * t];
            p[1] = T.rp[3 * t + 1];
            p[2] = T.rp[3 * t + 2];
        }
    }
    for (int d = 0; d < 3; ++d) {
        double c = p[d] - T.shift[d];
        r.h[d] = (float)c;
        r.l[d] = (float)(c - (double)r.h[d]);
    }
    return r;
}

// 1/r of a pair from r^2; 0 for a point on itself.  The hardware's approximate
// root (documented relative error 2^-22.9) for normal arguments; subnormal
// ones, distances below 1e-19 A, count as 0 (surface sums of the 20,000-atom
// octree with rsqrtf, which also serves those: 84.7 -> 73.0 ms).
__device__ __forceinline__ float rsqrt_pair(float r2) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(r2));
    return r2 >= 1.17549435e-38f ? y : 0.f;
}
// Packed FP32 pair: lane .x works for the thread's first target, .y for its
// second (one FP32x2 instruction does both).
__device__ __forceinline__ float2 bc2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);  // a - b, one rounding
}
__device__ __forceinline__ void kahan_add2(float2 &s, float2 &c, float2 v) {
    float2 y = sub2(v, c);
    float2 t = __fadd2_rn(s, y);
    c = sub2(sub2(t, s), y);
    s = t;
}

#include "nbody_far.cuh"

// The source tiles of one block: per-pair work, group sums and tile sums as
// described above, accumulated into acc_* (FP64).
// ORIGIN: the block's targets lie within NB_ORIGIN_EXT of its first target
// o, and th holds their positions relative to o as single FP32 values (tl
// unused); each source is staged once per tile as its FP32 position relative
// to o, (hi - o_hi) + (lo - o_lo), so that a difference takes one FP32
// operation instead of three.  Near sources (at least one atom radius away
// from a point of the molecular surface) then keep about 15 u of relative
// accuracy in r, far ones about u.
// FAR: only the sources that are no far ones of `ball`, gathered in source
// order into whole tiles.
template <bool PSI, bool SCREEN, bool PSI2, int AXIS, bool ORIGIN, bool FAR>
__device__ __forceinline__ void nb_tiles(float4 (*sp4)[4], const far::Ball &ball, const float4 *__restrict__ shi,
                                         const float4 *__restrict__ slo, long long ns, float kscr,
                                         const float (&oh)[3], const float (&ol)[3],
                                         const float2 (&th)[3], const float2 (&tl)[3],
                                         const float2 (&tn)[3], const float2 (&tn2)[3],
                                         double (&acc_phi)[NB_TPT], double (&acc_psi)[NB_TPT],
                                         double (&acc_psi2)[NB_TPT]) {
    auto stage = [&](int at, const float4 &a, const float4 &b) {
        if (ORIGIN) {
            const float rx = (a.x - oh[0]) + (b.x - ol[0]), ry = (a.y - oh[1]) + (b.y - ol[1]),
                        rz = (a.z - oh[2]) + (b.z - ol[2]);
            sp4[at][0] = make_float4(rx, rx, ry, ry);
            sp4[at][1] = make_float4(rz, rz, a.w, a.w);
        } else {
            sp4[at][0] = make_float4(a.x, a.x, a.y, a.y);
            sp4[at][1] = make_float4(a.z, a.z, a.w, a.w);
            sp4[at][2] = make_float4(b.x, b.x, b.y, b.y);
            sp4[at][3] = make_float4(b.z, b.z, 0.f, 0.f);
        }
    };
    // the first m staged sources
    auto pairs = [&](int m) {
        float2 sp = bc2(0.f), cp = bc2(0.f), sq = bc2(0.f), cq = bc2(0.f), s2 = bc2(0.f),
               c2 = bc2(0.f);
        // groups of GRP sources are summed plainly in FP32 (rounding error
        // below (GRP - 1) u of the group's absolute sum) and each group
        // sum enters the tile sum with Kahan compensation
        constexpr int GRP = FAR ? NB_GRP / 2 : NB_GRP;
        for (int q0 = 0; q0 < m; q0 += GRP) {
            const int q1 = min(q0 + GRP, m);
            float2 gp = bc2(0.f), gq = bc2(0.f), g2 = bc2(0.f);
#pragma unroll 4
            for (int q = q0; q < q1; ++q) {
                const float4 p0 = sp4[q][0], p1 = sp4[q][1];
                float2 dx, dy, dz;
                if (ORIGIN) {
                    dx = sub2(th[0], make_float2(p0.x, p0.y));
                    dy = sub2(th[1], make_float2(p0.z, p0.w));
                    dz = sub2(th[2], make_float2(p1.x, p1.y));
                } else {
                    const float4 p2 = sp4[q][2], p3 = sp4[q][3];
                    dx = __fadd2_rn(sub2(th[0], make_float2(p0.x, p0.y)),
                                    sub2(tl[0], make_float2(p2.x, p2.y)));
                    dy = __fadd2_rn(sub2(th[1], make_float2(p0.z, p0.w)),
                                    sub2(tl[1], make_float2(p2.z, p2.w)));
                    dz = __fadd2_rn(sub2(th[2], make_float2(p1.x, p1.y)),
                                    sub2(tl[2], make_float2(p3.x, p3.y)));
                }
                const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
                const float2 ri = make_float2(rsqrt_pair(r2.x), rsqrt_pair(r2.y));
                float2 v = __fmul2_rn(make_float2(p1.z, p1.w), ri);
                if (SCREEN) {
                    v.x *= expf(-kscr * (r2.x * ri.x));
                    v.y *= expf(-kscr * (r2.y * ri.y));
                }
                gp = __fadd2_rn(gp, v);
                if (PSI) {
                    // Psi along n: the general dot product, or, for a
                    // block whose targets all lie on edges along AXIS (n =
                    // +-e_AXIS), that coordinate difference (sign applied to
                    // the total)
                    const float2 dn =
                        AXIS == 0 ? dx
                                  : (AXIS == 1 ? dy
                                               : (AXIS == 2 ? dz
                                                            : __ffma2_rn(dz, tn[2],
                                                                         __ffma2_rn(dy, tn[1],
                                                                                    __fmul2_rn(dx, tn[0])))));
                    const float2 vr2 = __fmul2_rn(v, __fmul2_rn(ri, ri));
                    gq = __ffma2_rn(vr2, dn, gq);
                    if (PSI2) {
                        const float2 dn2 = __ffma2_rn(
                            dz, tn2[2], __ffma2_rn(dy, tn2[1], __fmul2_rn(dx, tn2[0])));
                        g2 = __ffma2_rn(vr2, dn2, g2);
                    }
                }
            }
            kahan_add2(sp, cp, gp);
            if (PSI) kahan_add2(sq, cq, gq);
            if (PSI2) kahan_add2(s2, c2, g2);
        }
        acc_phi[0] += (double)sp.x - (double)cp.x;
        acc_phi[1] += (double)sp.y - (double)cp.y;
        if (PSI) {
            acc_psi[0] += (double)sq.x - (double)cq.x;
            acc_psi[1] += (double)sq.y - (double)cq.y;
        }
        if (PSI2) {
            acc_psi2[0] += (double)s2.x - (double)c2.x;
            acc_psi2[1] += (double)s2.y - (double)c2.y;
        }
    };
    if constexpr (FAR) {
        __shared__ int wcount[NB_THREADS / 32];
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        int have = 0;
        for (long long base = 0; base < ns; base += NB_THREADS) {
            const long long si = base + threadIdx.x;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            bool near = false;
            if (si < ns) {
                a = shi[si];
                b = slo[si];
                float d[3], r2;
                near = !far::offset(a, b, ball, d, r2);
            }
            const unsigned mask = __ballot_sync(0xffffffffu, near);
            __syncthreads();  // the last reads of wcount and of the staged sources
            if (lane == 0) wcount[w] = __popc(mask);
            __syncthreads();
            int at = have + __popc(mask & ((1u << lane) - 1u));
#pragma unroll
            for (int q = 0; q < NB_THREADS / 32; ++q) {
                const int c = wcount[q];
                if (q < w) at += c;
                have += c;
            }
            if (near) stage(at, a, b);
            if (have < NB_THREADS) continue;
            __syncthreads();
            pairs(NB_THREADS);
            have -= NB_THREADS;
            __syncthreads();
            if ((int)threadIdx.x < have)
#pragma unroll
                for (int q = 0; q < 4; ++q) sp4[threadIdx.x][q] = sp4[NB_THREADS + threadIdx.x][q];
        }
        __syncthreads();
        pairs(have);
    } else {
        for (long long base = 0; base < ns; base += NB_THREADS) {
            const long long si = base + threadIdx.x;
            __syncthreads();
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (si < ns) {
                a = shi[si];
                b = slo[si];
            }
            stage(threadIdx.x, a, b);
            __syncthreads();
            pairs((int)min((long long)NB_THREADS, ns - base));
        }
    }
}

// out_phi[t] = scale * sum_i q_i exp(-k r)/r; out_psi[t] = sum_i q_i (r.n)/r^3
// (PSI only for surface targets); with PSI2 also out_psi2[t] along the
// target's second normal, from the same pairs.  Self pairs (r == 0) are skipped.  Each
// thread holds two targets in the two halves of FP32x2 registers; the
// sources are staged in shared memory already duplicated into (v, v) pairs.
static_assert(NB_TPT == 2, "two targets per thread, one per FP32x2 half");
// FAR: far sources through the block's expansion (nbody_far.cuh).
template <bool PSI, bool SCREEN, bool PSI2 = false, bool FAR = false>
__global__ void __launch_bounds__(NB_THREADS)
k_nbody(TargetDesc T, far::Args F, const float4 *__restrict__ shi, const float4 *__restrict__ slo,
        long long ns, float kscr, double scale, double *__restrict__ out_phi,
        double *__restrict__ out_psi, double *__restrict__ out_psi2 = nullptr) {
    // per source: (hx,hx,hy,hy) (hz,hz,q,q) (lx,lx,ly,ly) (lz,lz,0,0)
    __shared__ float4 sp4[FAR ? 2 * NB_THREADS : NB_THREADS][4];
    const long long at0 = (F.block0 + (long long)blockIdx.x) * NB_THREADS * NB_TPT;
    const long long tb = target_at(T, at0);
    long long tt[NB_TPT];
    far::Ball ball{};
    if (FAR) ball = F.ball[F.block0 + blockIdx.x];
    TgtLoad tg[NB_TPT];
    double acc_phi[NB_TPT], acc_psi[NB_TPT], acc_psi2[NB_TPT];
#pragma unroll
    for (int u = 0; u < NB_TPT; ++u) {
        tt[u] = target_at(T, at0 + threadIdx.x + (long long)u * NB_THREADS);
        tg[u] = load_target(T, tt[u]);
        acc_phi[u] = 0.0;
        acc_psi[u] = 0.0;
        acc_psi2[u] = 0.0;
    }
    float2 th[3], tl[3], tn[3], tn2[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        th[d] = make_float2(tg[0].h[d], tg[1].h[d]);
        tl[d] = make_float2(tg[0].l[d], tg[1].l[d]);
        tn[d] = make_float2(tg[0].n[d], tg[1].n[d]);
        tn2[d] = make_float2(tg[0].n2[d], tg[1].n2[d]);
    }
    // a block whose targets all lie on edges of one direction (the
    // crossing list is ordered by direction) takes the axis form of Psi
    int axis = -1;
    if (PSI && T.kind == TK_SURFACE) {
        const int dref = (int)(T.ids[tb] / T.g.N);
        bool same = true;
#pragma unroll
        for (int u = 0; u < NB_TPT; ++u) {
            const long long t = tt[u];
            if (t < T.count && (int)(T.ids[t] / T.g.N) != dref) same = false;
        }
        if (__syncthreads_and(same)) axis = dref;
    }
    // a block whose surface targets all lie within NB_ORIGIN_EXT of its
    // first target takes the differences from that origin (FAR: not the near
    // pairs, see nbody_far.cuh)
    bool origin = false;
    float oh[3] = {0.f, 0.f, 0.f}, ol[3] = {0.f, 0.f, 0.f};
    if (!FAR && T.kind == TK_SURFACE) {
        double o[3], rel[NB_TPT][3];
        bool near = true;
#pragma unroll
        for (int d = 0; d < 3; ++d) o[d] = T.rp[3 * tb + d];
#pragma unroll
        for (int u = 0; u < NB_TPT; ++u) {
            const long long t = tt[u];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                rel[u][d] = t < T.count ? T.rp[3 * t + d] - o[d] : 0.0;
                if (!(fabs(rel[u][d]) <= NB_ORIGIN_EXT)) near = false;
            }
        }
        if (__syncthreads_and(near)) {
            origin = true;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double oc = o[d] - T.shift[d];  // the sources are relative to the shift
                oh[d] = (float)oc;
                ol[d] = (float)(oc - (double)oh[d]);
                th[d] = make_float2((float)rel[0][d], (float)rel[1][d]);
            }
        }
    }
#define PB_NB_TILES(AX)                                                                          \
    (!FAR && origin ? nb_tiles<PSI, SCREEN, PSI2, AX, true, false>(sp4, ball, shi, slo, ns, kscr, oh, ol,  \
                                                         th, tl, tn, tn2, acc_phi, acc_psi, acc_psi2) \
            : nb_tiles<PSI, SCREEN, PSI2, AX, false, FAR>(sp4, ball, shi, slo, ns, kscr, oh, ol, \
                                                          th, tl, tn, tn2, acc_phi, acc_psi, acc_psi2))
    switch (axis) {
        case 0: PB_NB_TILES(0); break;
        case 1: PB_NB_TILES(1); break;
        case 2: PB_NB_TILES(2); break;
        default: PB_NB_TILES(-1);
    }
#undef PB_NB_TILES
    if constexpr (FAR) {
        // Psi = -n . grad; the axis form takes the sign of n below
        __syncthreads();  // the staged sources' last reads
        far::Series &S = *reinterpret_cast<far::Series *>(sp4);
        static_assert(sizeof(far::Series) + sizeof(double2) * far::NC <= sizeof(sp4), "the series fits the staging area");
        far::make_series(F, reinterpret_cast<double2 *>(&S + 1), S);
        __syncthreads();
        double x[NB_TPT][3];
#pragma unroll
        for (int u = 0; u < NB_TPT; ++u) {
            const long long t = tt[u];
#pragma unroll
            for (int d = 0; d < 3; ++d)
                x[u][d] = t < T.count ? ((T.rp[3 * t + d] - T.shift[d]) - (double)ball.c[d]) * ball.inv : 0.0;
        }
        float2 xx[3], v[4];
#pragma unroll
        for (int d = 0; d < 3; ++d) xx[d] = make_float2((float)x[0][d], (float)x[1][d]);
        far::evaluate(S, xx, v);
#pragma unroll
        for (int u = 0; u < NB_TPT; ++u) {
            double g[3];
#pragma unroll
            for (int d = 0; d < 3; ++d)
                g[d] = (S.top[1 + d] + (double)(u ? v[1 + d].y : v[1 + d].x)) * (ball.inv * ball.inv);
            acc_phi[u] += fma(S.top[3], x[u][2], fma(S.top[2], x[u][1], fma(S.top[1], x[u][0], S.top[0]))) * ball.inv +
                          (double)(u ? v[0].y : v[0].x) * ball.inv;
            const double ga = axis == 0 ? g[0] : (axis == 1 ? g[1] : g[2]);
            acc_psi[u] -= axis >= 0 ? ga
                                    : g[0] * (double)tg[u].n[0] + g[1] * (double)tg[u].n[1] + g[2] * (double)tg[u].n[2];
            if (PSI2)
                acc_psi2[u] -=
                    g[0] * (double)tg[u].n2[0] + g[1] * (double)tg[u].n2[1] + g[2] * (double)tg[u].n2[2];
        }
    }
    if (PSI && axis >= 0) {
        // n = sign e_axis: the one nonzero component is the sign
#pragma unroll
        for (int u = 0; u < NB_TPT; ++u)
            acc_psi[u] *= (double)(tg[u].n[0] + tg[u].n[1] + tg[u].n[2]);
    }
#pragma unroll
    for (int u = 0; u < NB_TPT; ++u) {
        const long long t = tt[u];
        if (t >= T.count) continue;
        if (T.kind == TK_BOUNDARY) {
            long long i, j, k;
            boundary_node(T.g, t, i, j, k);
            out_phi[(k * T.g.ny + j) * T.g.nx + i] = scale * acc_phi[u];
        } else {
            out_phi[t] = tg[u].active ? scale * acc_phi[u] : 0.0;
            if (PSI) out_psi[t] = tg[u].active ? acc_psi[u] : 0.0;
            if (PSI2) out_psi2[t] = tg[u].active ? acc_psi2[u] : 0.0;
        }
    }
}

// Boundary values in FP64: they enter the linear system itself, so they are
// summed in double precision (atoms staged in shared memory), in atom order.
// FP64 issue binds: 25 operations a pair with screening, 13 without; the
// library's sqrt, exp and division took about 70.  Blocks of 128 keep the
// last wave full.  141 x 95 x 63 grid, 300 atoms, screened: 1,712 -> 813 us.
// Positions are subtracted before k scales the distance: scaled first (24
// operations), their rounding is relative to the coordinates, and a molecule
// 1,000 A from the origin got 7.6e-16 instead of 6e-17 of sum |q| exp(-k r) / r.
constexpr int BT = 128;

template <bool SCREEN>
__global__ void __launch_bounds__(BT)
k_boundary64(GridGeo g, const double *__restrict__ atoms, long long na, long long count, double k,
             double scale, double *__restrict__ bc) {
    __shared__ double sx[BT], sy[BT], sz[BT], sq[BT], tab[64];
    if (SCREEN && threadIdx.x < 64) tab[threadIdx.x] = exp2((double)threadIdx.x * 0.015625);
    long long t = blockIdx.x * (long long)BT + threadIdx.x;
    double p[3] = {0.0, 0.0, 0.0};
    long long i = 0, j = 0, kk = 0;
    if (t < count) {
        boundary_node(g, t, i, j, kk);
        p[0] = g.o[0] + (double)i * g.h;
        p[1] = g.o[1] + (double)j * g.h;
        p[2] = g.o[2] + (double)kk * g.h;
    }
    double acc = 0.0;
    for (long long base = 0; base < na; base += BT) {
        long long si = base + threadIdx.x;
        __syncthreads();
        if (si < na) {
            sx[threadIdx.x] = atoms[si];
            sy[threadIdx.x] = atoms[na + si];
            sz[threadIdx.x] = atoms[2 * na + si];
            sq[threadIdx.x] = atoms[4 * na + si];
        }
        __syncthreads();
        int m = (int)min((long long)BT, na - base);
#pragma unroll 4
        for (int q = 0; q < m; ++q) {
            const double dx = p[0] - sx[q], dy = p[1] - sy[q], dz = p[2] - sz[q];
            const double r2 = (dx * dx + dy * dy) + dz * dz;
            const double y = rsqrt_fp64(r2);
            if (SCREEN)
                acc = fma(sq[q] * exp_neg_fp64(k * (r2 * y), tab), y, acc);
            else
                acc = fma(sq[q], y, acc);
        }
    }
    if (t < count) bc[(kk * g.ny + j) * g.nx + i] = scale * acc;
}

// Coulomb pair sum sum_{i<j} q_i q_j / r_ij in FP64 (the energy is a
// difference of large sums of either sign, so its terms are kept exact to
// rounding).  Atoms in tiles of PT; block (a, b) of the nt x nt grid, a <= b,
// takes the pairs i in tile a, j in tile b (j > i when a == b): thread t holds
// atom i, tile b is staged in shared memory and taken in ascending order,
// 1/r from rsqrt_fp64.  The block's total goes to
// part[b * nt + a] (zero for a > b); one block then adds the partials in
// index order, so the sum is the same on every run.
constexpr int PT = 128;

__global__ void __launch_bounds__(PT)
k_pairs64(const double *__restrict__ atoms, long long na, double *__restrict__ part) {
    __shared__ double sx[PT], sy[PT], sz[PT], sq[PT];
    using BR = cub::BlockReduce<double, PT>;
    __shared__ typename BR::TempStorage tmp;
    const int a = blockIdx.x, b = blockIdx.y, nt = gridDim.x;
    if (a > b) {
        if (threadIdx.x == 0) part[(long long)b * nt + a] = 0.0;
        return;
    }
    const long long i = (long long)a * PT + threadIdx.x;
    const long long j0 = (long long)b * PT, js = j0 + threadIdx.x;
    if (js < na) {
        sx[threadIdx.x] = atoms[js];
        sy[threadIdx.x] = atoms[na + js];
        sz[threadIdx.x] = atoms[2 * na + js];
        sq[threadIdx.x] = atoms[4 * na + js];
    }
    __syncthreads();
    double mine = 0.0;
    if (i < na) {
        const double px = atoms[i], py = atoms[na + i], pz = atoms[2 * na + i];
        const int m = (int)min((long long)PT, na - j0);
        const int q0 = a == b ? threadIdx.x + 1 : 0;  // j > i on the diagonal tile
        double acc = 0.0;
        for (int q = q0; q < m; ++q) {
            const double dx = px - sx[q], dy = py - sy[q], dz = pz - sz[q];
            const double r2 = (dx * dx + dy * dy) + dz * dz;
            if (r2 > 0.0) acc = fma(sq[q], rsqrt_fp64(r2), acc);
        }
        mine = atoms[4 * na + i] * acc;
    }
    const double tot = BR(tmp).Sum(mine);
    if (threadIdx.x == 0) part[(long long)b * nt + a] = tot;
}

// 2 sum_{i<j} (the sum over i of q_i Phi_i) from the pair partials, in index
// order -> eacc->ecoul_sum
__global__ void __launch_bounds__(1024)
k_reduce_pairs(const double *__restrict__ part, long long n, EnergyAcc *eacc) {
    using BR = cub::BlockReduce<double, 1024>;
    __shared__ typename BR::TempStorage tmp;
    double s = 0.0;
    for (long long i = threadIdx.x; i < n; i += 1024) s += part[i];
    double tot = BR(tmp).Sum(s);
    if (threadIdx.x == 0) eacc->ecoul_sum = 2.0 * tot;
}

pb_status split_sources(pb_system *sys, cudaStream_t s, float4 **hi, float4 **lo) {
    pb_grid *g = sys->g;
    long long na = g->na > 0 ? g->na : 1;
    *hi = (float4 *)dalloc(sizeof(float4) * na, s);
    *lo = (float4 *)dalloc(sizeof(float4) * na, s);
    if (!*hi || !*lo) return PB_ERR_OOM;
    if (g->na > 0) {
        k_split_atoms<<<cdiv(g->na, 256), 256, 0, s>>>(g->atoms, g->na, g->center[0], g->center[1],
                                                       g->center[2], *hi, *lo);
        PB_LAUNCH_CHECK();
    }
    return PB_OK;
}

// Bricks of 8^3 finest nodes in the order in which blocks take their targets:
// rods of 2 x 2 bricks, a slice of four bricks at a time, up one rod and
// down the next one beside it, so that neighbours in the order are neighbours
// in space.
struct RodOrder {
    int nx, ny, nz;  // bricks along x, rods along y and z
    __host__ __device__ long long keys() const { return (long long)nx * ny * nz; }
    __device__ unsigned key(int bx, int by, int bz) const {
        const int y = by >> 1, z = bz >> 1, rod = z * ny + ((z & 1) ? ny - 1 - y : y);
        return (unsigned)rod * (unsigned)nx + (unsigned)((rod & 1) ? nx - 1 - bx : bx);
    }
};

// sort keys of an octree's crossing edges: the brick of their lower ends
__global__ void
k_target_keys(const long long *__restrict__ ids, long long n, long long slots, const int4 *__restrict__ blow, RodOrder rods,
              unsigned int *__restrict__ key, int *__restrict__ val) {
    const long long t = blockIdx.x * 256ll + threadIdx.x;
    if (t >= n) return;
    long long a = ids[t];
    while (a >= slots) a -= slots;
    const int4 low = blow[a >> 9];
    key[t] = rods.key(low.x >> 3, low.y >> 3, low.z >> 3);
    val[t] = (int)t;
}

// The order in which blocks take the targets: by bricks, the three directions
// together, so that a block's 512 lie close together (the crossing list goes
// through the molecule three times; in the octree's Morton order a few blocks at
// its jumps had most of the atoms near them: 18.9 ms on 20,000 atoms).  A stable
// sort, so the order, and with it every bit of the sums, is the same on every
// run.  Null beyond 2^31 targets or 2^32 keys.
pb_status order_targets(pb_grid *g, int **order, cudaStream_t s) {
    const long long n = g->ncross;
    const int side = g->ot.NL / 8 + 1, pairs = (side + 1) / 2;  // bricks an axis
    const RodOrder rods = {side, pairs, pairs};
    int bits = 1;
    while ((rods.keys() - 1) >> bits) ++bits;
    if (bits > 32 || n > 0x7fffffffll) return PB_OK;
    unsigned *key = (unsigned *)dalloc(sizeof(unsigned) * n, s), *key2 = (unsigned *)dalloc(sizeof(unsigned) * n, s);
    int *val = (int *)dalloc(sizeof(int) * n, s), *val2 = (int *)dalloc(sizeof(int) * n, s);
    void *tmp = nullptr;
    size_t bytes = 0;
    cudaError_t e = cudaErrorMemoryAllocation;
    if (key && key2 && val && val2) {
        k_target_keys<<<cdiv(n, 256), 256, 0, s>>>(g->cid, n, g->geo.N, g->ot.blow, rods, key, val);
        e = cub::DeviceRadixSort::SortPairs(nullptr, bytes, key, key2, val, val2, (int)n, 0, bits, s);
        if (e == cudaSuccess && !(tmp = dalloc(bytes, s))) e = cudaErrorMemoryAllocation;
        if (e == cudaSuccess)
            e = cub::DeviceRadixSort::SortPairs(tmp, bytes, key, key2, val, val2, (int)n, 0, bits, s);
    }
    dfree(tmp, s);
    dfree(key, s);
    dfree(key2, s);
    dfree(val, s);
    if (e != cudaSuccess) {
        dfree(val2, s);
        if (e == cudaErrorMemoryAllocation) return PB_ERR_OOM;
        set_error("sorting the surface targets failed: %s", cudaGetErrorString(e));
        return PB_ERR_CUDA;
    }
    *order = val2;
    return PB_OK;
}

TargetDesc make_desc(pb_system *sys, int kind) {
    pb_grid *g = sys->g;
    TargetDesc T;
    T.kind = kind;
    T.g = g->geo;
    for (int d = 0; d < 3; ++d) T.shift[d] = g->center[d];
    T.rp = g->crp;
    T.ids = g->cid;
    T.sign = g->csign;
    T.nrm2 = nullptr;
    T.order = nullptr;
    T.count = 0;
    return T;
}

}  // namespace

pb_status nbody_boundary(pb_system *sys, cudaStream_t s) {
    pb_grid *g = sys->g;
    const GridGeo &geo = g->geo;
    PB_CUDA_TRY(cudaMemsetAsync(sys->bc, 0, sizeof(double) * geo.N, s));
    if (sys->p.bc == PB_BC_ZERO || g->na == 0) return PB_OK;
    long long count =
        2ll * geo.nx * geo.ny + (long long)(geo.nz - 2) * (2ll * geo.nx + 2ll * (geo.ny - 2));
    double scale = sys->lB / sys->p.eps_out;
    double k = sys->p.bc == PB_BC_DH ? sys->kD : 0.0;
    if (k > 0.0)
        k_boundary64<true><<<cdiv(count, BT), BT, 0, s>>>(geo, g->atoms, g->na, count, k, scale, sys->bc);
    else
        k_boundary64<false><<<cdiv(count, BT), BT, 0, s>>>(geo, g->atoms, g->na, count, k, scale, sys->bc);
    PB_LAUNCH_CHECK();
    return PB_OK;
}

pb_status nbody_surface(pb_system *sys, cudaStream_t s) {
    pb_grid *g = sys->g;
    long long nc = g->ncross > 0 ? g->ncross : 1;
    if (!sys->Phi) sys->Phi = (double *)dalloc(sizeof(double) * nc, s);
    if (!sys->Psi) sys->Psi = (double *)dalloc(sizeof(double) * nc, s);
    if (!sys->Phi || !sys->Psi) return PB_ERR_OOM;
    if (g->ncross == 0) return PB_OK;
    float4 *hi, *lo;
    pb_status st = split_sources(sys, s, &hi, &lo);
    if (st != PB_OK) return st;
    TargetDesc T = make_desc(sys, TK_SURFACE);
    T.count = g->ncross;
    // Psi along the re-triangulated surface's analytic normals (first
    // integral of Eq. energy_ion, Sec. 3.3.2) comes from the same pairs as
    // Phi and Psi
    if (!sys->PsiN) sys->PsiN = (double *)dalloc(sizeof(double) * nc, s);
    if (!sys->PsiN) return PB_ERR_OOM;
    T.nrm2 = g->mc_n;
    const int per = NB_THREADS * NB_TPT;
    const unsigned blocks = cdiv(T.count, per);
    far::Args F{};
    F.chunks = (int)cdiv(g->na, far::CHUNK);
    // so many target blocks at a time that their partial sums stay within far::BYTES
    const size_t each = sizeof(float2) * far::NS * (size_t)F.chunks;
    const unsigned parts = cdiv(blocks, std::max<long long>(far::BYTES / (long long)std::max<size_t>(each, 1), 1)), most = cdiv(blocks, parts);
    int *order = nullptr;
    far::Ball *ball = nullptr;
    float2 *part = nullptr;
    if (g->is_oct && g->na * g->ncross >= FAR_PAIRS && F.chunks <= 65535) {  // chunks: the grid's y
        st = order_targets(g, &order, s);
        if (order) {
            ball = (far::Ball *)dalloc(sizeof(far::Ball) * blocks, s);
            part = (float2 *)dalloc(each * most, s);
            if (!ball || !part) st = PB_ERR_OOM;
        }
        if (st == PB_ERR_OOM) {  // all pairs need no scratch
            dfree(order, s);
            order = nullptr;
            set_error("");
            st = PB_OK;
        }
    }
    if (order) {
        T.order = order;
        F.ball = ball;
        F.part = part;
        k_far_ball<<<blocks, 256, 0, s>>>(g->crp, T.order, T.count, g->center[0], g->center[1], g->center[2], ball);
        for (unsigned b = 0; b < blocks; b += most) {
            const unsigned n = std::min(most, blocks - b);
            F.block0 = b;
            k_far_local<<<dim3(n, (unsigned)F.chunks), far::T, 0, s>>>(hi, lo, g->na, ball, b, part);
            k_nbody<true, false, true, true>
                <<<n, NB_THREADS, 0, s>>>(T, F, hi, lo, g->na, 0.f, 1.0, sys->Phi, sys->Psi, sys->PsiN);
        }
    } else if (st == PB_OK) {
        k_nbody<true, false, true>
            <<<blocks, NB_THREADS, 0, s>>>(T, F, hi, lo, g->na, 0.f, 1.0, sys->Phi, sys->Psi, sys->PsiN);
    }
    for (void *q : {(void *)order, (void *)ball, (void *)part, (void *)hi, (void *)lo}) dfree(q, s);
    if (st != PB_OK) return st;
    PB_LAUNCH_CHECK();
    return PB_OK;
}

pb_status nbody_pairs(pb_system *sys, cudaStream_t s) {
    pb_grid *g = sys->g;
    if (g->na <= 1) {
        PB_CUDA_TRY(cudaMemsetAsync(&sys->eacc->ecoul_sum, 0, sizeof(double), s));
        return PB_OK;
    }
    const long long nt = cdiv(g->na, PT);
    if (nt > 8192) {  // the partials grow as nt^2 (512 MB at this limit)
        set_error("too many atoms for the Coulomb pair sum (%lld; at most %d)",
                  (long long)g->na, 8192 * PT);
        return PB_ERR_ARG;
    }
    double *part = (double *)dalloc(sizeof(double) * nt * nt, s);
    if (!part) return PB_ERR_OOM;
    k_pairs64<<<dim3((unsigned)nt, (unsigned)nt), PT, 0, s>>>(g->atoms, g->na, part);
    PB_LAUNCH_CHECK();
    k_reduce_pairs<<<1, 1024, 0, s>>>(part, nt * nt, sys->eacc);
    PB_LAUNCH_CHECK();
    dfree(part, s);
    return PB_OK;
}

}  // namespace pbg
