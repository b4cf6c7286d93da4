// Far atoms of the surface sums by local expansions (included by nbody.cu).
//
// A block's targets (512 neighbours of the crossing list) lie in a ball of
// radius a.  Atoms further than KAPPA a from its centre c act on all of them
// through one expansion in solid harmonics about c, in a unit of about a:
//   sum_i q_i / |x - y_i| = sum_{l <= P} sum_m R_lm(x) conj(L_lm),
//   L_lm = sum_i q_i I_lm(y_i),
//   R_lm = r^l P_lm e^{im phi} / (l + m)!,  I_lm = (l - m)! P_lm e^{im phi} / r^(l+1)
// (addition theorem of the Legendre polynomials, no Condon-Shortley phase), by
//   R_mm = (x + iy) R_{m-1,m-1} / 2m,  (l+m)(l-m) R_lm = (2l-1) z R_{l-1,m} - r^2 R_{l-2,m},
//   I_mm = (2m-1)(x + iy) I_{m-1,m-1} / r^2,
//   I_lm = [(2l-1) z I_{l-1,m} - ((l-1)^2 - m^2) I_{l-2,m}] / r^2.
// The gradient is a series in the same R_lm of degree P - 1, from
//   d/dz R_lm = R_{l-1,m},  (d/dx -+ i d/dy) R_lm = +-R_{l-1,m-+1}.
// The nearer atoms are summed pair by pair, with the split differences: from a
// block's origin (one FP32 operation) their error is larger, and it showed where
// all pairs had no such blocks (9,000 atoms at 0.5 A: Psi 2.02e-7 from 64
// bits against 1.69e-7; split 1.55e-7, in the same time).
//
// P = 12 and KAPPA = 3 leave a truncation error below one FP32 rounding of
// sum |q| / r^2 in the gradient (at most 4.2e-8 in blocks at the surface of
// 20,000 atoms in a 45 A ball, a = 3 and 5 A, against 64 bits; P = 11: 9.5e-8)
// and 2.8e-10 of sum |q| / r in the potential, below the rounding of the FP32
// pair sum.  Atoms beyond 2 KAPPA a take degree PD.
//
// Measured (GB300, surface sums, all pairs -> this): octree of 20,000 atoms
// 73.0 -> 8.7 ms (coefficients 4.5, near pairs and evaluation 3.9), 2,000
// atoms 0.9 -> 0.53 ms.  Errors against 64 bits,
// 2-norm relative, of Phi 1.26e-7 -> 8.1e-8 and of Psi 1.84e-7 -> 1.53e-7 (20,000
// atoms).  What gave it, one after the other: targets in list order, whose
// blocks are wide, 20.6 ms; a power of two as unit and compensated sums of
// degrees 0 and 1, no slower and more exact than all pairs; rods of bricks as
// order 10.9 ms; the lower degree for distant atoms 8.7 ms.
#pragma once

namespace far {

constexpr int P = 12, NC = (P + 1) * (P + 2) / 2;  // coefficients with m >= 0, by columns of m
constexpr float KAPPA = 3.f;
constexpr int PD = 8;        // degree for atoms beyond 2 KAPPA a: (2 KAPPA)^-(PD + 1) < KAPPA^-(P + 1)
constexpr int T = 128;       // threads of k_far_local: 64 atoms at a time, half of the columns a thread
constexpr int CHUNK = 2048;  // atoms of a partial sum: 32 in a row a thread
constexpr long long BYTES = 32ll << 20;  // of the partial sums of one pair of launches, at most

__host__ __device__ constexpr int at(int l, int m) { return m * (P + 1) - m * (m - 1) / 2 + l - m; }
// the columns of the first half; 46 coefficients against 45
__host__ __device__ constexpr bool first_half(int m) { return (m & 3) == 0 || (m & 3) == 3; }

struct Ball {
    float c[3];         // relative to the sources' shift
    float r2far;        // (KAPPA a)^2
    double inv;         // 1 / unit of length: the power of two next above a, so that scaling is exact
};

// offset of a source from the ball's centre, and whether it is a far one (the
// same operations wherever it is asked)
__device__ __forceinline__ bool offset(const float4 &a, const float4 &b, const Ball &ball, float (&d)[3], float &r2) {
    d[0] = __fadd_rn(__fsub_rn(a.x, ball.c[0]), b.x);
    d[1] = __fadd_rn(__fsub_rn(a.y, ball.c[1]), b.y);
    d[2] = __fadd_rn(__fsub_rn(a.z, ball.c[2]), b.z);
    r2 = __fmaf_rn(d[2], d[2], __fmaf_rn(d[1], d[1], __fmul_rn(d[0], d[0])));
    return r2 > ball.r2far;
}

struct Args {
    const Ball *ball;    // of every target block
    const float2 *part;  // partial L of the launch's blocks: [block][chunk][NS]
    int chunks;
    unsigned block0;     // first target block of the launch
};

}  // namespace far

// Balls of the target blocks, two targets a thread
__global__ void __launch_bounds__(256)
k_far_ball(const double *__restrict__ rp, const int *__restrict__ order, long long count, double sx, double sy, double sz,
           far::Ball *__restrict__ ball) {
    __shared__ float red[8][6];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double shift[3] = {sx, sy, sz};
    double p[2][3];
    float v[6];  // -min, max
    for (int u = 0; u < 2; ++u) {
        // places past the list repeat its last target
        const long long t = order[min((long long)blockIdx.x * 512 + u * 256 + threadIdx.x, count - 1)];
        for (int d = 0; d < 3; ++d) {
            p[u][d] = rp[3 * t + d] - shift[d];
            const float x = (float)p[u][d];
            v[d] = u ? fmaxf(v[d], -x) : -x;
            v[3 + d] = u ? fmaxf(v[3 + d], x) : x;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < 6; ++q) v[q] = fmaxf(v[q], __shfl_xor_sync(0xffffffffu, v[q], o));
    if (lane == 0)
        for (int q = 0; q < 6; ++q) red[w][q] = v[q];
    __syncthreads();
    for (int q = 0; q < 6; ++q)
        for (int r = 0; r < 8; ++r) v[q] = fmaxf(v[q], red[r][q]);
    __syncthreads();
    float c[3], r2 = 0.f;
    for (int d = 0; d < 3; ++d) c[d] = 0.5f * (v[3 + d] - v[d]);
    for (int u = 0; u < 2; ++u) {
        const float x = (float)(p[u][0] - (double)c[0]), y = (float)(p[u][1] - (double)c[1]),
                    z = (float)(p[u][2] - (double)c[2]);
        r2 = fmaxf(r2, (x * x + y * y) + z * z);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
    if (lane == 0) red[w][0] = r2;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int r = 1; r < 8; ++r) r2 = fmaxf(r2, red[r][0]);
    far::Ball &b = ball[blockIdx.x];
    const float a = fmaxf(1.00001f * sqrtf(r2), 0.25f);
    for (int d = 0; d < 3; ++d) b.c[d] = c[d];
    b.r2far = (far::KAPPA * a) * (far::KAPPA * a);
    int e;
    frexpf(a, &e);
    b.inv = ldexp(1.0, -e);
}

namespace far {
// first place of column m among the sums of its half
__host__ __device__ constexpr int place(int m) {
    int k = 0;
    for (int q = 0; q < m; ++q)
        if (first_half(q) == first_half(m)) k += P + 1 - q;
    return k;
}
constexpr int HALF = 46;
// The coefficients of degree 0 and 1 carry most of a sum: they are summed with
// compensation, and their partial sums are FP32 pairs (the second parts after
// the NC first ones).
constexpr int NS = NC + 3;
__host__ __device__ constexpr int low(int l, int m) { return l == 0 ? 0 : 1 + m; }  // place of a second part

// adds q I_lm(d), l <= D, of columns M .. D of one half to acc; mm: q I_M-1,M-1
template <int M, bool FIRST, int D>
__device__ __forceinline__ void add_irregular(float2 mm, const float2 &e, float zr, float ir2, float2 (&acc)[HALF],
                                              float2 (&comp)[2]) {
    if constexpr (M > 0) {
        const float ex = (float)(2 * M - 1) * e.x, ey = (float)(2 * M - 1) * e.y;
        mm = make_float2(ex * mm.x - ey * mm.y, ex * mm.y + ey * mm.x);
    }
    if constexpr (first_half(M) == FIRST) {
        constexpr int K = place(M);
        float2 b = make_float2(0.f, 0.f), a = mm;  // degrees l - 1 and l
        if (M <= 1) kahan_add2(acc[K], comp[0], a);
        else acc[K] = __fadd2_rn(acc[K], a);
#pragma unroll
        for (int j = 1; j <= D - M; ++j) {
            const int l = M + j;
            const float cz = (float)(2 * l - 1) * zr, cb = -(float)((l - 1) * (l - 1) - M * M) * ir2;
            const float2 n = j == 1 ? __fmul2_rn(make_float2(cz, cz), a)
                                    : __ffma2_rn(make_float2(cz, cz), a, __fmul2_rn(make_float2(cb, cb), b));
            b = a;
            a = n;
            if (l <= 1) kahan_add2(acc[K + j], comp[1], a);
            else acc[K + j] = __fadd2_rn(acc[K + j], a);
        }
    }
    if constexpr (M < D) add_irregular<M + 1, FIRST, D>(mm, e, zr, ir2, acc, comp);
}

// the warp's totals of columns M .. P of one half
template <int M, bool FIRST>
__device__ __forceinline__ void warp_totals(const float2 (&acc)[HALF], const float2 (&comp)[2], float2 *red,
                                            double2 *exact) {
    if constexpr (first_half(M) == FIRST) {
#pragma unroll
        for (int j = 0; j <= P - M; ++j) {
            float2 v = acc[place(M) + j];
            if (M + j <= 1) {
                double2 x = make_double2((double)v.x - (double)comp[j].x, (double)v.y - (double)comp[j].y);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    x.x += __shfl_xor_sync(0xffffffffu, x.x, o);
                    x.y += __shfl_xor_sync(0xffffffffu, x.y, o);
                }
                if ((threadIdx.x & 31) == 0) exact[low(M + j, M)] = x;
                continue;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
                v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
            }
            if ((threadIdx.x & 31) == 0) red[at(M + j, M)] = v;
        }
    }
    if constexpr (M < P) warp_totals<M + 1, FIRST>(acc, comp, red, exact);
}

// the n listed sources of a chunk, 64 at a time
template <bool FIRST, int D>
__device__ __forceinline__ void add_list(const float4 *shi, const float4 *slo, const uint16_t *list, int n, const Ball &ball,
                                         float2 (&acc)[HALF], float2 (&comp)[2]) {
    const float inv = (float)ball.inv;
    for (int k = threadIdx.x & (T / 2 - 1); k < n; k += T / 2) {
        const int i = list[k];
        const float4 a = shi[i];
        float d[3], r2;
        offset(a, slo[i], ball, d, r2);
        // 1/r with one Newton step: an error here is one of all targets
        const float x = inv * d[0], y = inv * d[1], z = inv * d[2], s2 = inv * inv * r2, r0 = rsqrtf(s2);
        const float ri = __fmaf_rn(0.5f * r0, __fmaf_rn(-(s2 * r0), r0, 1.f), r0), ir2 = ri * ri;
        add_irregular<0, FIRST, D>(make_float2(a.w * ri, 0.f), make_float2(x * ir2, y * ir2), z * ir2, ir2, acc, comp);
    }
}

template <bool FIRST>
__device__ __forceinline__ void local(const float4 *shi, const float4 *slo, const uint16_t *mid, int nmid,
                                      const uint16_t *distant, int ndistant, const Ball &ball, float2 (*red)[NC],
                                      double2 (*exact)[3]) {
    float2 acc[HALF], comp[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int k = 0; k < HALF; ++k) acc[k] = make_float2(0.f, 0.f);
    add_list<FIRST, P>(shi, slo, mid, nmid, ball, acc, comp);
    add_list<FIRST, PD>(shi, slo, distant, ndistant, ball, acc, comp);
    __syncwarp();
    const int w = (threadIdx.x >> 5) & 1;
    warp_totals<0, FIRST>(acc, comp, red[w], exact[w]);
}
}  // namespace far

// Partial L_lm of one target block (x) and one chunk of the sources (y).
// Bound by FP32 issue: about 300 (degree P) or 160 (degree PD) instructions a
// source and half of the columns, against 8,000 for its 512 pairs.  All
// coefficients in one thread would take 182 registers of sums.
__global__ void __launch_bounds__(far::T, 3)
k_far_local(const float4 *__restrict__ shi, const float4 *__restrict__ slo, long long ns,
            const far::Ball *__restrict__ ball, unsigned block0, float2 *__restrict__ part) {
    using namespace far;
    __shared__ float2 red[2][NC];
    __shared__ double2 exact[2][3];
    const Ball b = ball[block0 + blockIdx.x];
    const long long s0 = (long long)blockIdx.y * CHUNK, s1 = min(s0 + CHUNK, ns);
    // the chunk's far sources by the degree that they take, in order
    __shared__ uint16_t mid[CHUNK], distant[CHUNK];
    __shared__ int counts[T / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, n = (int)(s1 - s0);
    const unsigned below = (1u << lane) - 1u;
    shi += s0;
    slo += s0;
    int nm = 0, nd = 0;
    for (int base = 0; base < n; base += T) {
        const int i = base + threadIdx.x;
        float d[3], r2 = 0.f;
        const bool is = i < n && offset(shi[i], slo[i], b, d, r2), deg = is && r2 <= 4.f * b.r2far;
        const unsigned bm = __ballot_sync(0xffffffffu, deg), bd = __ballot_sync(0xffffffffu, is && !deg);
        __syncthreads();
        if (lane == 0) counts[w] = __popc(bm) | (__popc(bd) << 16);
        __syncthreads();
        int am = nm + __popc(bm & below), ad = nd + __popc(bd & below);
#pragma unroll
        for (int q = 0; q < T / 32; ++q) {
            const int c = counts[q];
            if (q < w) {
                am += c & 0xffff;
                ad += c >> 16;
            }
            nm += c & 0xffff;
            nd += c >> 16;
        }
        if (deg) mid[am] = (uint16_t)i;
        else if (is) distant[ad] = (uint16_t)i;
    }
    __syncthreads();
    if (threadIdx.x < T / 2) local<true>(shi, slo, mid, nm, distant, nd, b, red, exact);
    else local<false>(shi, slo, mid, nm, distant, nd, b, red, exact);
    __syncthreads();
    float2 *out = part + ((long long)blockIdx.x * gridDim.y + blockIdx.y) * NS;
    for (int k = threadIdx.x; k < NC; k += T)
        if (k > 1 && k != at(1, 1)) out[k] = make_float2(red[0][k].x + red[1][k].x, red[0][k].y + red[1][k].y);
    if (threadIdx.x < 3) {
        const int q = threadIdx.x;
        const double x = exact[0][q].x + exact[1][q].x, y = exact[0][q].y + exact[1][q].y;
        const float2 h = make_float2((float)x, (float)y);
        out[q < 2 ? q : at(1, 1)] = h;
        out[NC + q] = make_float2((float)(x - (double)h.x), (float)(y - (double)h.y));
    }
}

namespace far {
// The block's expansion in shared memory: for every (l, m) the coefficients of
// the potential and of its three derivatives, each value twice (a thread's two
// targets share an instruction), 2 for m > 0 included; those of R_00, which
// are the largest, apart in FP64 (the gradient's are the potential's linear
// term too: with charges of one sign that is a tenth of the potential).
struct Series {
    float4 c[NC][4];  // potential, d/dx, d/dy, d/dz: (re, re, im, im)
    double top[4];
};
// L: NC pairs of scratch
__device__ __forceinline__ void make_series(const Args &A, double2 *L, Series &S) {
    const float2 *p = A.part + (long long)blockIdx.x * A.chunks * NS;
    for (int k = threadIdx.x; k < NC; k += blockDim.x) {
        double2 s = make_double2(0.0, 0.0);
        const int lo = k <= 1 ? NC + k : (k == at(1, 1) ? NC + 2 : -1);
        for (int c = 0; c < A.chunks; ++c) {
            const float2 v = p[(long long)c * NS + k];
            s.x += (double)v.x;
            s.y += (double)v.y;
            if (lo >= 0) {
                const float2 r = p[(long long)c * NS + lo];
                s.x += (double)r.x;
                s.y += (double)r.y;
            }
        }
        L[k] = s;
    }
    __syncthreads();
    for (int m = 0; m <= P; ++m) {
        const int l = m + threadIdx.x;
        if (l > P) continue;
        auto get = [&](int l, int m) {  // L_l,-m = (-1)^m conj L_lm
            if (m >= 0) return L[at(l, m)];
            const double2 v = L[at(l, -m)];
            return (m & 1) ? make_double2(-v.x, v.y) : make_double2(v.x, -v.y);
        };
        const double w = m ? 2.0 : 1.0;
        double2 v[4] = {get(l, m), {0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
        if (l < P) {
            const double2 u = get(l + 1, m + 1), d = get(l + 1, m - 1);
            v[1] = make_double2(0.5 * (u.x - d.x), 0.5 * (u.y - d.y));
            v[2] = make_double2(0.5 * (u.y + d.y), -0.5 * (u.x + d.x));
            v[3] = get(l + 1, m);
        }
        for (int q = 0; q < 4; ++q) {
            const float re = (float)(w * v[q].x), im = (float)(w * v[q].y);
            S.c[at(l, m)][q] = make_float4(re, re, im, im);
            if (l == 0) S.top[q] = v[q].x;
        }
    }
}
// potential (without its terms of degrees 0 and 1, top[0] + top[1..3] . x) and
// gradient (without those of degree 0, top[1..3]) at two targets, in the ball's unit
__device__ __forceinline__ void evaluate(const Series &S, const float2 (&x)[3], float2 (&out)[4]) {
    const float2 one = make_float2(1.f, 1.f), r2 = __ffma2_rn(x[2], x[2], __ffma2_rn(x[1], x[1], __fmul2_rn(x[0], x[0])));
    const float2 nr2 = make_float2(-r2.x, -r2.y), ny = make_float2(-x[1].x, -x[1].y);
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q] = make_float2(0.f, 0.f);
    float2 mr = one, mi = make_float2(0.f, 0.f);  // R_mm
#pragma unroll
    for (int m = 0; m <= P; ++m) {
        if (m > 0) {
            const float s = 1.f / (float)(2 * m);
            const float2 ss = make_float2(s, s);
            const float2 re = __fmul2_rn(ss, __ffma2_rn(x[0], mr, __fmul2_rn(ny, mi)));
            mi = __fmul2_rn(ss, __ffma2_rn(x[0], mi, __fmul2_rn(x[1], mr)));
            mr = re;
        }
        float2 ar = mr, ai = mi, br = make_float2(0.f, 0.f), bi = br;
#pragma unroll
        for (int l = m; l <= P; ++l) {
            if (l > m) {
                const float s = 1.f / (float)((l + m) * (l - m)), z = (float)(2 * l - 1) * s;
                const float2 cz = __fmul2_rn(make_float2(z, z), x[2]), cb = __fmul2_rn(make_float2(s, s), nr2);
                const float2 nr = __ffma2_rn(cz, ar, __fmul2_rn(cb, br)), ni = __ffma2_rn(cz, ai, __fmul2_rn(cb, bi));
                br = ar;
                bi = ai;
                ar = nr;
                ai = ni;
            }
            if (l == 0) continue;
#pragma unroll
            for (int q = l == 1 ? 1 : 0; q < 4; ++q) {
                const float4 v = S.c[at(l, m)][q];
                out[q] = __ffma2_rn(make_float2(v.x, v.y), ar, __ffma2_rn(make_float2(v.z, v.w), ai, out[q]));
            }
        }
    }
}
}  // namespace far
