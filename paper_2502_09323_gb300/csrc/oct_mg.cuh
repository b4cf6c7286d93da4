// Two-level preconditioner of the octree's FP32 PCG (included by octree.cu).
//
// The trilinear functions of the uniform lattice at the coarsest spacing are a
// subspace of the octree's functions, so one lattice serves as coarse space
// whatever the refinement: z = smoothing, lattice correction, smoothing.  The
// lattice problem takes one V-cycle (mg.cuh), on edge weights averaged from
// the finest lattice (unrefined regions are solvent).  The lattice is 2^Lmax
// times coarser than the finest cells, so the smoother is a Chebyshev
// polynomial in D^-1 A on [2/a, 2] (A is an M-matrix with non-negative row
// sums, so its largest eigenvalue is at most 2); degree 2, a = 10 for two
// levels of refinement.  Prototype on the CPU, iterations to 1e-6: 60 atoms
// 269 (Jacobi) -> 13, 200 atoms 374 -> 14; three levels (degree 3, a = 20)
// 298 -> 15.  More levels keep the Jacobi preconditioner.
//
// Measured (GB300, 20,000 atoms, 41.7M unknowns): 1,341 -> 32 iterations to
// 1e-12, the solve 685 -> 71 ms; an iteration takes 1.9 ms (steps 263 and 270
// us, residual 220, prolongation 145, partial sums 82, gather 37, V-cycle on
// 145^3 110, direction and update kernels 236 and 268).
//
// A step of the polynomial is one pass of the brick kernel
//   x_k+1 = x_k + a_k (x_k - x_k-1) + b_k (s - D^-1 A x_k),  s = D^-1 r.
// The residual is restricted in two steps without atomics: every brick sums
// its nodes onto the lattice nodes of its closed box, then every lattice node
// adds the sums of the bricks around it in a fixed order.
#pragma once

constexpr int OMG_LMAX = 3;     // levels of refinement at most
constexpr int OMG_PART = 128;   // lattice nodes of a refined brick (125, 27, 8) in its partials

__host__ __device__ constexpr int omg_side(int level) { return 8 >> level; }  // lattice cells of a brick's side

// Residual (per slot) of the refined bricks summed onto their lattice nodes.
// Four bricks a block, 64 threads each; a dimension at a time.
__global__ void __launch_bounds__(OB) k_omg_partial(OctDev t, const float *__restrict__ r, float *__restrict__ part,
                                                    const CgState *st) {
    if (*(volatile const int *)&st->done) return;
    __shared__ float A[4][5][64], B[4][5][5][8];
    const int g = threadIdx.x >> 6, c = threadIdx.x & 63;
    for (long long b0 = (long long)blockIdx.x * 4; b0 < t.nb; b0 += (long long)gridDim.x * 4) {
        const long long b = b0 + g;
        const int level = b < t.nb ? t.blow[b].w : 0;
        const int n = omg_side(level), m = 1 << level;  // lattice cells, nodes per cell
        const float inv = 1.f / (float)m;
        const bool act = b < t.nb && level > 0;
        __syncthreads();
        if (act) {  // row (j, k) along x
            const float4 *p = reinterpret_cast<const float4 *>(r + (b << 9) + 8 * c);
            const float4 u = p[0], v = p[1];
            const float x[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
            float carry = 0.f;
            for (int q = 0; q <= n; ++q) {
                float s = carry;
                carry = 0.f;
                if (q < n)
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if ((i >> level) == q) {
                            const float f = (float)(i & (m - 1)) * inv;
                            s += (1.f - f) * x[i];
                            carry += f * x[i];
                        }
                A[g][q][c] = s;
            }
        }
        __syncthreads();
        if (act)
            for (int o = c; o < (n + 1) * 8; o += 64) {  // (x node, plane k) along y
                const int q = o >> 3, k = o & 7;
                float carry = 0.f;
                for (int w = 0; w <= n; ++w) {
                    float s = carry;
                    carry = 0.f;
                    if (w < n)
                        for (int i = 0; i < m; ++i) {
                            const float f = (float)i * inv, v = A[g][q][8 * k + w * m + i];
                            s += (1.f - f) * v;
                            carry += f * v;
                        }
                    B[g][w][q][k] = s;
                }
            }
        __syncthreads();
        if (act)
            for (int o = c; o < (n + 1) * (n + 1); o += 64) {  // (x, y node) along z
                const int w = o / (n + 1), q = o - w * (n + 1);
                float carry = 0.f;
                for (int u = 0; u <= n; ++u) {
                    float s = carry;
                    carry = 0.f;
                    if (u < n)
                        for (int i = 0; i < m; ++i) {
                            const float f = (float)i * inv, v = B[g][w][q][u * m + i];
                            s += (1.f - f) * v;
                            carry += f * v;
                        }
                    part[b * OMG_PART + (u * (n + 1) + w) * (n + 1) + q] = s;
                }
            }
    }
}

// s = D^-1 (sum over the bricks around a lattice node), interior nodes
__global__ void __launch_bounds__(256) k_omg_gather(OctDev t, const float *__restrict__ r, const float *__restrict__ part,
                                                    LatticeMg L, const CgState *st) {
    if (*(volatile const int *)&st->done) return;
    const int m = L.n - 2;
    const long long a = blockIdx.x * 256ll + threadIdx.x;
    if (a >= (long long)m * m * m) return;
    const int X[3] = {1 + (int)(a % m), 1 + (int)((a / m) % m), 1 + (int)(a / ((long long)m * m))};
    const int s0 = 1 << t.Lmax;
    int br[8];
    float sum = 0.f;
#pragma unroll
    for (int o = 0; o < 8; ++o) {
        // the lattice cell on this side lies in one finest-brick cell
        const int cx = ((X[0] - 1 + (o & 1)) * s0) >> 3, cy = ((X[1] - 1 + ((o >> 1) & 1)) * s0) >> 3,
                  cz = ((X[2] - 1 + (o >> 2)) * s0) >> 3;
        const int b = t.bmap[cidx(t, cx, cy, cz)];
        br[o] = b;
        bool seen = false;
        for (int q = 0; q < o; ++q) seen = seen || br[q] == b;
        if (seen) continue;
        const int4 low = t.blow[b];
        const int lx = X[0] - (low.x >> t.Lmax), ly = X[1] - (low.y >> t.Lmax), lz = X[2] - (low.z >> t.Lmax);
        if (low.w == 0) {  // its own nodes are lattice nodes
            if (lx < 8 && ly < 8 && lz < 8) sum += r[((long long)b << 9) + (lz * 8 + ly) * 8 + lx];
        } else {
            const int n = omg_side(low.w) + 1;
            sum += part[(long long)b * OMG_PART + (lz * n + ly) * n + lx];
        }
    }
    const int p = X[2] * L.sxy + X[1] * L.sx + X[0];
    L.s[p] = __fdividef(sum, __ldg(L.dg + p));
}

// x += P e on the unknowns.  Four bricks a block; a refined brick's lattice
// values are staged in shared memory.
__global__ void __launch_bounds__(OB) k_omg_prolong(OctDev t, const uint8_t *__restrict__ code, LatticeMg L,
                                                    float *__restrict__ x, const CgState *st) {
    if (*(volatile const int *)&st->done) return;
    __shared__ float E[4][125];
    const int g = threadIdx.x >> 6, c = threadIdx.x & 63;
    for (long long b0 = (long long)blockIdx.x * 4; b0 < t.nb; b0 += (long long)gridDim.x * 4) {
        const long long b = b0 + g;
        const bool act = b < t.nb;
        const int4 low = act ? t.blow[b] : make_int4(0, 0, 0, 0);
        const int level = low.w, n = omg_side(level) + 1, m = 1 << level;
        const int p0 = (low.z >> t.Lmax) * L.sxy + (low.y >> t.Lmax) * L.sx + (low.x >> t.Lmax);
        __syncthreads();
        if (act && level > 0)
            for (int q = c; q < n * n * n; q += 64) {
                const int lx = q % n, ly = (q / n) % n, lz = q / (n * n);
                E[g][q] = L.z[p0 + lz * L.sxy + ly * L.sx + lx];
            }
        __syncthreads();
        if (!act) continue;
        const int i = c & 7, j = c >> 3;
        const float inv = 1.f / (float)m;
        const int ci = i >> level, cj = j >> level;
        const float fx = (float)(i & (m - 1)) * inv, fy = (float)(j & (m - 1)) * inv;
        // the value at (i, j) of lattice plane u of the brick
        auto plane = [&](int u) {
            const float *e = &E[g][(u * n + cj) * n + ci];
            const float a0 = e[0] + fx * (e[1] - e[0]), a1 = e[n] + fx * (e[n + 1] - e[n]);
            return a0 + fy * (a1 - a0);
        };
        float ea = 0.f, eb = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float e;
            if (level == 0) {
                e = L.z[p0 + k * L.sxy + j * L.sx + i];
            } else {
                if ((k & (m - 1)) == 0) {
                    ea = k == 0 ? plane(0) : eb;
                    eb = plane((k >> level) + 1);
                }
                e = ea + (float)(k & (m - 1)) * inv * (eb - ea);
            }
            const long long a = (b << 9) + 64 * k + c;
            const int kind = code[a] >> 4;
            if (kind == 0 || kind == 3) x[a] += e;
        }
    }
}

// Weights and ionic term of the lattice at twice the finest spacing, averaged
// from the finest lattice as k_mg_coarsen does (mean of the harmonic and the
// arithmetic combination along an edge, the weights of P^T across).  Outside
// the finest bricks the finest weights are the solvent's.  n nodes an axis,
// rows of sx.
__global__ void __launch_bounds__(128)
k_omg_lattice(OctDev t, const double *__restrict__ W0, const double *__restrict__ W1, const double *__restrict__ W2,
              const uint8_t *__restrict__ inside, float w_out, float kap_out, int n, int sx, float *__restrict__ wx,
              float *__restrict__ wy, float *__restrict__ wz, float *__restrict__ kap) {
    const long long a = blockIdx.x * 128ll + threadIdx.x;
    if (a >= (long long)n * n * n) return;
    const int X[3] = {(int)(a % n), (int)((a / n) % n), (int)(a / ((long long)n * n))};
    const long long p = ((long long)X[2] * n + X[1]) * sx + X[0];
    const int last = t.NL;  // finest nodes 0 .. NL
    // the eight finest-brick cells that the fine nodes 2 X - 1 .. 2 X + 2 lie in
    int lo[3], hi[3];
    bool pure = true;
    for (int d = 0; d < 3; ++d) {
        lo[d] = max(2 * X[d] - 1, 0) >> 3;
        hi[d] = min(min(2 * X[d] + 2, last) >> 3, t.nf - 1);
        lo[d] = min(lo[d], t.nf - 1);
    }
    for (int q = 0; q < 8; ++q)
        pure = pure && t.lev[cidx(t, (q & 1) ? hi[0] : lo[0], (q & 2) ? hi[1] : lo[1], (q & 4) ? hi[2] : lo[2])] != t.Lmax;
    const bool ex[3] = {X[0] < n - 1, X[1] < n - 1, X[2] < n - 1};
    if (pure) {
        wx[p] = ex[0] ? 2.f * w_out : 0.f;
        wy[p] = ex[1] ? 2.f * w_out : 0.f;
        wz[p] = ex[2] ? 2.f * w_out : 0.f;
        kap[p] = 8.f * kap_out;
        return;
    }
    auto slot = [&](int x, int y, int z) -> long long {  // of a finest-level node, else -1
        if (x >= last || y >= last || z >= last) return -1;
        const long long c = cidx(t, x >> 3, y >> 3, z >> 3);
        if (t.lev[c] != t.Lmax) return -1;
        return ((long long)t.bmap[c] << 9) + (((z & 7) * 8 + (y & 7)) * 8 + (x & 7));
    };
    const double *W[3] = {W0, W1, W2};
    float out[3];
    for (int d = 0; d < 3; ++d) {
        const int u = (d + 1) % 3, v = (d + 2) % 3;
        float sum = 0.f;
        for (int b = -1; b <= 1; ++b)
            for (int c = -1; c <= 1; ++c) {
                int x[3];
                x[u] = min(max(2 * X[u] + c, 0), last);
                x[v] = min(max(2 * X[v] + b, 0), last);
                x[d] = 2 * X[d];
                long long m = slot(x[0], x[1], x[2]);
                const float f = m >= 0 ? (float)W[d][m] : w_out;
                x[d] += 1;
                m = slot(x[0], x[1], x[2]);
                const float g = m >= 0 ? (float)W[d][m] : w_out;
                sum += (b ? 0.5f : 1.f) * (c ? 0.5f : 1.f) * 0.5f * (f * (g / (f + g)) + 0.25f * (f + g));
            }
        out[d] = ex[d] ? sum : 0.f;
    }
    float ks = 0.f;
    for (int e = 0; e < 27; ++e) {
        const int x = e % 3 - 1, y = (e / 3) % 3 - 1, z = e / 9 - 1;
        const long long m = slot(min(max(2 * X[0] + x, 0), last), min(max(2 * X[1] + y, 0), last),
                                 min(max(2 * X[2] + z, 0), last));
        ks += (x ? 0.5f : 1.f) * (y ? 0.5f : 1.f) * (z ? 0.5f : 1.f) * (m >= 0 && inside[m] ? 0.f : kap_out);
    }
    wx[p] = out[0];
    wy[p] = out[1];
    wz[p] = out[2];
    kap[p] = ks;
}

// the polynomial: steps x_k+1 from x_k, x_k-1 and s
struct OmgStep {
    float a, b;
};
struct OmgPoly {
    int degree;
    float first;         // x_1 = first * s from x_0 = 0
    OmgStep step[8];     // step k: a_k, b_k (step 0: a = 0, b = first)
};
inline OmgPoly omg_poly(int Lmax) {
    OmgPoly P{};
    P.degree = Lmax >= 3 ? 3 : 2;
    const double hi = 2.0, lo = hi / (Lmax >= 3 ? 20.0 : 10.0);
    const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), sigma = theta / delta;
    P.first = (float)(1.0 / theta);
    P.step[0] = {0.f, P.first};
    double rho = 1.0 / sigma;
    for (int k = 1; k < P.degree; ++k) {
        const double r = 1.0 / (2.0 * sigma - rho);
        P.step[k] = {(float)(r * rho), (float)(2.0 * r / delta)};
        rho = r;
    }
    return P;
}
