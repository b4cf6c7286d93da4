// Multigrid preconditioner of the FP32 PCG (included by solve.cu).
//
// One V(1,1) cycle of damped Jacobi on a hierarchy of vertex-centred grids
// replaces the Jacobi preconditioner z = D^-1 r of the FP32 inner solve: a
// symmetric positive definite preconditioner, so the PCG around it is the
// same recurrence.  Coarse node I is fine node 2 I; a coarse grid has
// n/2 + 1 nodes an axis, its last node a boundary node (one spacing past
// the fine boundary when n - 1 is odd: the last coarse edge is then half as
// long).  Trilinear interpolation P, restriction P^T.  A coarse edge weight
// is, along the edge, the mean of the harmonic and the arithmetic
// combination of the two fine edges, summed across with the weights of P^T;
// the ionic term is summed with the weights of P^T.  Measured on the CPU
// (129^3, 1,000 atoms, eps 2/80): 14 iterations to 1e-6 against 290 with
// Jacobi, and harmonic or arithmetic alone 15.
//
// Every level keeps s = D^-1 b (b its right-hand side) instead of b, so that
// all levels share one pair of kernels:
//   down:  r = b - A (w s) = (1 - w) d s + w sum_f W_f s_f ;
//          s_coarse = D_c^-1 P^T r
//   up:    v = w s + P z_coarse ; z = (1 - w) v + w (s + D^-1 sum_f W_f v_f)
// Level 0 uses the compressed operator (code bytes and listed weights), the
// coarse levels a float4 (W+x, W+y, W+z, diagonal) per node.  The levels
// whose data fits one block's shared memory are solved by one block per
// system in one launch (k_mg_bottom).  The up kernel of level 0 also sums
// rho = r.z and takes the CG step beta = rho / rho_old.
//
// Measured (GB300, solves to 1e-12): 257^3 155.6 -> 20.5 ms (1,127 -> 30
// iterations), 65^3 30.6 -> 3.8 ms, a batch of 24 systems of 97^3 to 161^3
// 229 -> 71 ms.
//
// Bounds: down reads s and a code byte per fine node and writes an eighth of
// a value; up reads s, an eighth of a value and a code byte and writes z.
#pragma once

namespace mg {

constexpr int LMAX = 12;            // levels at most
constexpr float OMEGA = 0.85f;      // Jacobi damping (0.8 to 0.9 take the same iterations)
constexpr int NT = 256;
constexpr int BOT_T = 1024;         // threads of the bottom kernel
constexpr int BOT_NODES = 7300;     // nodes of all its levels (28 B each in shared memory)
constexpr int SWEEPS = 8;           // Jacobi sweeps on the coarsest level
constexpr int FX = 64, FY = 16;     // fine nodes of a block's tile
constexpr int CX = FX / 2, CY = FY / 2;

struct Lev {
    int nx, ny, nz, sx, sxy;
    float *s, *z;                   // D^-1 b, solution (level 0: the solver's z32 and v32)
    float4 *cf;                     // W+x, W+y, W+z, diagonal (levels >= 1)
};

// One system (device memory, or the kernel parameter of a one-system launch)
struct Entry {
    Lev lev[LMAX];
    int nlev, nbot;                 // levels; first level of the bottom kernel
    int dbase[LMAX], ubase[LMAX];   // first work item of this system in a level's launches
    int dk[LMAX], uk[LMAX];         // planes per work item (coarse planes down, fine planes up)
    CgState *st;
    const uint8_t *code;
    CoefC32 cp;
    float *partials;                // rho of each work item of the level-0 up kernel
    int nu0;                        // their number
};

// launch totals of a table, read on the device
struct Head {
    int nsys;
    unsigned int done;              // blocks finished (level-0 up kernel)
    int dtotal[LMAX], utotal[LMAX];
};

__host__ __device__ inline int ditems(const Entry &e, int l) {
    if (l >= e.nbot) return 0;
    const Lev &c = e.lev[l + 1];
    return ((c.nx - 1 + CX - 1) / CX) * ((c.ny - 1 + CY - 1) / CY) * ((c.nz - 2 + e.dk[l] - 1) / e.dk[l]);
}
__host__ __device__ inline int uitems(const Entry &e, int l) {
    if (l >= e.nbot) return 0;
    const Lev &f = e.lev[l];
    return ((f.nx - 1 + FX - 1) / FX) * ((f.ny - 1 + FY - 1) / FY) * ((f.nz - 2 + e.uk[l] - 1) / e.uk[l]);
}

// sum over the six faces of W x_neighbour, and the diagonal
template <bool FINE>
__device__ __forceinline__ float face_sum(const Entry &e, const Lev &L, int p, float xm, float xp, float ym,
                                          float yp, float zm, float zp, float &d) {
    if constexpr (FINE) {
        const uint32_t c = e.code[p];
        const uint32_t cx = e.code[p - 1], cy = e.code[p - L.sx], cz = e.code[p - L.sxy];
        const float w = (c & 1) ? e.cp.w_in : e.cp.w_out;
        const float kap = (c & 1) ? 0.f : e.cp.kap;
        if (((c & 0xEu) | (cx & 2u) | (cy & 4u) | (cz & 8u)) == 0u) {
            d = 6.f * w + kap;
            return w * (((xm + xp) + (ym + yp)) + (zm + zp));
        }
        const float w0 = (cx & 2u) ? __ldg(e.cp.wx + p - 1) : w;
        const float w1 = (c & 2u) ? __ldg(e.cp.wx + p) : w;
        const float w2 = (cy & 4u) ? __ldg(e.cp.wy + p - L.sx) : w;
        const float w3 = (c & 4u) ? __ldg(e.cp.wy + p) : w;
        const float w4 = (cz & 8u) ? __ldg(e.cp.wz + p - L.sxy) : w;
        const float w5 = (c & 8u) ? __ldg(e.cp.wz + p) : w;
        d = (((((w0 + w1) + w2) + w3) + w4) + w5) + kap;
        return ((w0 * xm + w1 * xp) + (w2 * ym + w3 * yp)) + (w4 * zm + w5 * zp);
    } else {
        const float4 q = __ldg(L.cf + p);
        const float w0 = __ldg(&L.cf[p - 1].x), w2 = __ldg(&L.cf[p - L.sx].y), w4 = __ldg(&L.cf[p - L.sxy].z);
        d = q.w;
        return ((w0 * xm + q.x * xp) + (w2 * ym + q.y * yp)) + (w4 * zm + q.z * zp);
    }
}

__device__ __forceinline__ bool interior(const Lev &L, int i, int j, int k) {
    return i >= 1 && j >= 1 && k >= 1 && i <= L.nx - 2 && j <= L.ny - 2 && k <= L.nz - 2;
}

// the system of a work item
__device__ __forceinline__ int find_sys(const Entry *tab, int nsys, int it, int (Entry::*base)[LMAX], int l) {
    int lo = 0, hi = nsys - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((tab[mid].*base)[l] <= it) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

}  // namespace mg

// Residual after the pre-smoothing step and its restriction.  A block takes
// CX x CY coarse nodes and marches over its coarse planes; the fine s of four
// planes and the residual of two are in shared memory, so that one barrier
// a fine plane suffices; a plane's loads are issued one plane ahead.
template <bool FINE, bool SINGLE>
__global__ void __launch_bounds__(mg::NT, 5)
k_mg_down(const mg::Entry *__restrict__ tab, const mg::Head *__restrict__ head, int l, int total,
          const __grid_constant__ mg::Entry e0) {
    using namespace mg;
    constexpr int SW = FX + 4, SH = FY + 4, RW = FX + 1, RH = FY + 1;
    constexpr int NLD = (SW / 2 * SH + NT - 1) / NT;
    __shared__ float sp[4][SH][SW];
    __shared__ float rb[2][RH][RW + 1];
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int nsys = SINGLE ? 1 : head->nsys;
    if (!SINGLE) total = head->dtotal[l];
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        const Entry &e = SINGLE ? e0 : tab[find_sys(tab, nsys, it, &Entry::dbase, l)];
        if (*(volatile int *)&e.st->done) continue;
        const Lev L = e.lev[l], C = e.lev[l + 1];
        const int li = SINGLE ? it : it - e.dbase[l];
        const int xt = (C.nx - 1 + CX - 1) / CX, yt = (C.ny - 1 + CY - 1) / CY;
        const int col = li % (xt * yt), ch = li / (xt * yt);
        const int i0 = (col % xt) * FX, j0 = (col / xt) * FY;
        const int K0 = 1 + ch * e.dk[l], K1 = min(K0 + e.dk[l], C.nz - 1);
        const int ka = 2 * K0 - 1, kb = 2 * K1 - 1;  // fine planes ka .. kb of the residual
        float2 ld[NLD];
        auto load = [&](int k) {
#pragma unroll
            for (int q = 0; q < NLD; ++q) {
                const int t = tid + q * NT, r = t / (SW / 2), c = t - r * (SW / 2);
                const int i = i0 - 2 + 2 * c, j = j0 - 2 + r;
                ld[q] = make_float2(0.f, 0.f);
                if (t < SW / 2 * SH && i >= 0 && i < L.sx && j >= 0 && j < L.ny && k >= 0 && k < L.nz)
                    ld[q] = *reinterpret_cast<const float2 *>(L.s + (k * L.sxy + j * L.sx + i));
            }
        };
        auto store = [&](int k) {
#pragma unroll
            for (int q = 0; q < NLD; ++q) {
                const int t = tid + q * NT, r = t / (SW / 2), c = t - r * (SW / 2);
                if (t < SW / 2 * SH) *reinterpret_cast<float2 *>(&sp[k & 3][r][2 * c]) = ld[q];
            }
        };
        __syncthreads();  // the previous item's last reads
        load(ka - 1);
        store(ka - 1);
        load(ka);
        store(ka);
        load(ka + 1);
        float acc = 0.f;
        for (int k = ka; k <= kb + 1; ++k) {
            if (k <= kb) store(k + 1);
            __syncthreads();
            if (k < kb) load(k + 2);
            if (k <= kb) {
                const float (*sm)[SW] = sp[(k - 1) & 3], (*sc)[SW] = sp[k & 3], (*sn)[SW] = sp[(k + 1) & 3];
                const int pk = k * L.sxy;
#pragma unroll
                for (int q = 0; q < (RW * RH + NT - 1) / NT; ++q) {
                    const int t = tid + q * NT, r = t / RW, c = t - r * RW;
                    if (t < RW * RH) {
                        const int i = i0 - 1 + c, j = j0 - 1 + r;
                        float v = 0.f;
                        if (interior(L, i, j, k)) {
                            float d;
                            const float s0 = sc[r + 1][c + 1];
                            const float sum = face_sum<FINE>(e, L, pk + j * L.sx + i, sc[r + 1][c], sc[r + 1][c + 2],
                                                             sc[r][c + 1], sc[r + 2][c + 1], sm[r + 1][c + 1],
                                                             sn[r + 1][c + 1], d);
                            v = (1.f - OMEGA) * d * s0 + OMEGA * sum;
                        }
                        rb[k & 1][r][c] = v;
                    }
                }
            }
            if (k > ka) {  // restrict plane k - 1
                const float (*b)[RW + 1] = rb[(k - 1) & 1];
                float t = 0.f;
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    const float *row = &b[2 * ty + r][2 * tx];
                    const float x = row[1] + 0.5f * (row[0] + row[2]);
                    t += r == 1 ? x : 0.5f * x;
                }
                if ((k - 1) & 1) {
                    acc += 0.5f * t;
                    const int K = (k - 2) >> 1, I = i0 / 2 + tx, J = j0 / 2 + ty;
                    if (k - 1 > ka && interior(C, I, J, K)) {
                        const int pc = K * C.sxy + J * C.sx + I;
                        C.s[pc] = __fdividef(acc, __ldg(&C.cf[pc].w));
                    }
                    acc = 0.5f * t;
                } else {
                    acc += t;
                }
            }
        }
    }
}

// Interpolated correction, post-smoothing step and (level 0) rho = r.z.  A
// block takes FX x FY fine nodes and marches over its fine planes; v, s and
// the coarse correction of four planes each are in shared memory.
template <bool FINE, bool SINGLE>
__global__ void __launch_bounds__(mg::NT, 4)
k_mg_up(const mg::Entry *__restrict__ tab, mg::Head *__restrict__ head, int l, int total,
        const __grid_constant__ mg::Entry e0) {
    using namespace mg;
    constexpr int VW = FX + 2, VH = FY + 2, EW = CX + 2, EH = CY + 2;
    constexpr int NV = (VW * VH + NT - 1) / NT, NE = (EW * EH + NT - 1) / NT;
    __shared__ float vp[4][VH][VW];
    __shared__ float ss[4][VH][VW];
    __shared__ float ec[4][EH][EW];
    __shared__ float sred[NT / 32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int nsys = SINGLE ? 1 : head->nsys;
    if (!SINGLE) total = head->utotal[l];
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        const Entry &e = SINGLE ? e0 : tab[find_sys(tab, nsys, it, &Entry::ubase, l)];
        if (*(volatile int *)&e.st->done) continue;
        const Lev L = e.lev[l], C = e.lev[l + 1];
        const int li = SINGLE ? it : it - e.ubase[l];
        const int xt = (L.nx - 1 + FX - 1) / FX, yt = (L.ny - 1 + FY - 1) / FY;
        const int col = li % (xt * yt), ch = li / (xt * yt);
        const int i0 = (col % xt) * FX, j0 = (col / xt) * FY;
        const int k0 = 1 + ch * e.uk[l], k1 = min(k0 + e.uk[l], L.nz - 1);
        float lds[NV], lde[NE];
        auto load_s = [&](int k) {
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const int t = tid + q * NT, r = t / VW, c = t - r * VW;
                const int i = i0 - 1 + c, j = j0 - 1 + r;
                lds[q] = 0.f;
                if (t < VW * VH && interior(L, i, j, k)) lds[q] = L.s[k * L.sxy + j * L.sx + i];
            }
        };
        auto load_e = [&](int K) {
#pragma unroll
            for (int q = 0; q < NE; ++q) {
                const int t = tid + q * NT, r = t / EW, c = t - r * EW;
                const int I = i0 / 2 - 1 + c, J = j0 / 2 - 1 + r;
                lde[q] = 0.f;
                if (t < EW * EH && interior(C, I, J, K)) lde[q] = C.z[K * C.sxy + J * C.sx + I];
            }
        };
        auto store_e = [&](int K) {
#pragma unroll
            for (int q = 0; q < NE; ++q) {
                const int t = tid + q * NT, r = t / EW, c = t - r * EW;
                if (t < EW * EH) ec[K & 3][r][c] = lde[q];
            }
        };
        // v = w s + P e of plane k
        auto make_v = [&](int k) {
            const float (*ea)[EW] = ec[(k >> 1) & 3], (*eb)[EW] = ec[((k + 1) >> 1) & 3];
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const int t = tid + q * NT, r = t / VW, c = t - r * VW;
                if (t < VW * VH) {
                    const int i = i0 - 1 + c, j = j0 - 1 + r;
                    float v = 0.f;
                    if (interior(L, i, j, k)) {
                        // coarse columns and rows either side (the same one on a coarse line)
                        const int a = (c + 1) >> 1, b = (c + 2) >> 1, m = (r + 1) >> 1, n = (r + 2) >> 1;
                        const float x = (ea[m][a] + ea[m][b]) + (ea[n][a] + ea[n][b]);
                        const float y = (eb[m][a] + eb[m][b]) + (eb[n][a] + eb[n][b]);
                        v = OMEGA * lds[q] + 0.125f * (x + y);
                    }
                    vp[k & 3][r][c] = v;
                    ss[k & 3][r][c] = lds[q];
                }
            }
        };
        __syncthreads();  // the previous item's last reads
        for (int K = (k0 - 1) >> 1; K <= (k0 + 2) >> 1; ++K) {
            load_e(K);
            store_e(K);
        }
        __syncthreads();
        load_s(k0 - 1);
        make_v(k0 - 1);
        load_s(k0);
        make_v(k0);
        load_s(k0 + 1);
        // coarse planes up to (k0 + 2) / 2 are here: those of v(k0 + 1)
        float rho = 0.f;
        for (int k = k0; k < k1; ++k) {
            float s0[4];
            make_v(k + 1);
            // the coarse plane that v(k + 2) needs anew
            const int Kn = (k + 3) >> 1;
            const bool fresh = (k + 2) & 1;
            if (fresh) load_e(Kn);
            load_s(k + 2);
            if (fresh) store_e(Kn);
            __syncthreads();
            const float (*vm)[VW] = vp[(k - 1) & 3], (*vc)[VW] = vp[k & 3], (*vn)[VW] = vp[(k + 1) & 3];
            const int pk = k * L.sxy;
#pragma unroll
            for (int q = 0; q < FX * FY / NT; ++q) {
                const int t = tid + q * NT, r = 1 + t / FX, c = 1 + t % FX;
                const int i = i0 - 1 + c, j = j0 - 1 + r;
                s0[q] = ss[k & 3][r][c];
                if (interior(L, i, j, k)) {
                    const int p = pk + j * L.sx + i;
                    float d;
                    const float sum = face_sum<FINE>(e, L, p, vc[r][c - 1], vc[r][c + 1], vc[r - 1][c], vc[r + 1][c],
                                                     vm[r][c], vn[r][c], d);
                    const float z = (1.f - OMEGA) * vc[r][c] + OMEGA * (s0[q] + __fdividef(sum, d));
                    L.z[p] = z;
                    if (FINE) rho += d * s0[q] * z;
                }
            }
        }
        if (FINE) {
            rho = tma::warp_sum_f(rho);
            if (lane == 0) sred[w] = rho;
            __syncthreads();
            if (tid == 0) {
                float t = 0.f;
                for (int q = 0; q < NT / 32; ++q) t += sred[q];
                e.partials[li] = t;
            }
        }
    }
    if (!FINE) return;
    // the last block sums every system's items in item order and takes the
    // CG step: beta = rho / rho_old
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&head->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    auto finish = [&](CgState *st, double t) {
        if (st->done) return;
        if (!(t > 0.0) || !isfinite(t)) {
            st->done = 1;
            st->status = 1;
            return;
        }
        st->beta = st->rho > 0.0 ? t / st->rho : 0.0;
        st->rho = t;
    };
    constexpr int BIG = 256;
    __shared__ double dred[NT / 32];
    for (int q = 0; q < nsys; ++q) {
        const Entry &e = SINGLE ? e0 : tab[q];
        const int n = e.nu0;
        if (n <= BIG || *(volatile int *)&e.st->done) continue;
        float s = 0.f, c = 0.f;
#pragma unroll 4
        for (int i = tid; i < n; i += NT) tma::nsum(s, c, __ldcg(e.partials + i));
        tma::warp_nsum(s, c);
        if (lane == 0) dred[w] = (double)s + (double)c;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int r = 0; r < NT / 32; ++r) t += dred[r];
            finish(e.st, t);
        }
        __syncthreads();
    }
    for (int q = w; q < nsys; q += NT / 32) {
        const Entry &e = SINGLE ? e0 : tab[q];
        const int n = e.nu0;
        if (n == 0 || n > BIG || *(volatile int *)&e.st->done) continue;
        float s = 0.f, c = 0.f;
#pragma unroll 4
        for (int i = lane; i < n; i += 32) tma::nsum(s, c, __ldcg(e.partials + i));
        tma::warp_nsum(s, c);
        if (lane == 0) finish(e.st, (double)s + (double)c);
    }
    if (tid == 0) head->done = 0u;
}

// The levels nbot .. nlev - 1 of one system per block, in shared memory.
// The same cycle as above; SWEEPS damped Jacobi steps on the last level.
template <bool SINGLE>
__global__ void __launch_bounds__(mg::BOT_T, 1)
k_mg_bottom(const mg::Entry *__restrict__ tab, const mg::Head *__restrict__ head,
            const __grid_constant__ mg::Entry e0) {
    using namespace mg;
    extern __shared__ __align__(16) float4 bsm[];
    const int tid = threadIdx.x;
    if (!SINGLE) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!SINGLE && (int)blockIdx.x >= head->nsys) return;
    const Entry &e = SINGLE ? e0 : tab[blockIdx.x];
    const int lb = e.nbot, le = e.nlev;
    if (le == 0) return;
    // the coefficients do not depend on the previous kernel
    int off = 0;
    for (int l = lb; l < le; ++l) {
        const Lev &L = e.lev[l];
        const int n = L.sxy * L.nz;
        for (int p = tid; p < n; p += BOT_T) bsm[off + p] = __ldg(L.cf + p);
        off += n;
    }
    float *S = reinterpret_cast<float *>(bsm + off), *Z = S + off, *R = Z + off;
    for (int p = tid; p < off; p += BOT_T) S[p] = Z[p] = R[p] = 0.f;
    if (SINGLE) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*(volatile int *)&e.st->done) return;
    __syncthreads();
    {
        const Lev &L = e.lev[lb];
        const int n = L.sxy * L.nz;
        for (int p = tid; p < n; p += BOT_T) S[p] = L.s[p];
    }
    __syncthreads();
    // sum over the faces of node p of a level whose coefficients start at cf
    auto faces = [&](const float4 *cf, const Lev &L, const float *x, int p) {
        const float4 q = cf[p];
        return ((cf[p - 1].x * x[p - 1] + q.x * x[p + 1]) + (cf[p - L.sx].y * x[p - L.sx] + q.y * x[p + L.sx])) +
               (cf[p - L.sxy].z * x[p - L.sxy] + q.z * x[p + L.sxy]);
    };
    auto each = [&](const Lev &L, auto f) {  // interior nodes
        const int mx = L.nx - 2, my = L.ny - 2, m = mx * my * (L.nz - 2);
        for (int t = tid; t < m; t += BOT_T) {
            const int r = t / mx, i = 1 + t - r * mx, k = 1 + r / my, j = 1 + r - (r / my) * my;
            f(i, j, k, k * L.sxy + j * L.sx + i);
        }
    };
    int o = 0;
    for (int l = lb; l < le - 1; ++l) {
        const Lev &L = e.lev[l], &C = e.lev[l + 1];
        const int oc = o + L.sxy * L.nz;
        each(L, [&](int, int, int, int p) {
            R[o + p] = (1.f - OMEGA) * bsm[o + p].w * S[o + p] + OMEGA * faces(bsm + o, L, S + o, p);
        });
        __syncthreads();
        each(C, [&](int I, int J, int K, int pc) {
            float acc = 0.f;
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const float *x = R + o + (2 * K - 1 + c) * L.sxy + (2 * J - 1 + b) * L.sx + 2 * I;
                    const float t = x[0] + 0.5f * (x[-1] + x[1]);
                    acc += (b == 1 ? 1.f : 0.5f) * (c == 1 ? 1.f : 0.5f) * t;
                }
            S[oc + pc] = __fdividef(acc, bsm[oc + pc].w);
        });
        __syncthreads();
        o = oc;
    }
    {
        const Lev &L = e.lev[le - 1];
        float *a = Z + o, *b = R + o;
        each(L, [&](int, int, int, int p) { a[p] = OMEGA * S[o + p]; });
        __syncthreads();
        for (int q = 1; q < SWEEPS; ++q) {
            each(L, [&](int, int, int, int p) {
                b[p] = (1.f - OMEGA) * a[p] + OMEGA * (S[o + p] + __fdividef(faces(bsm + o, L, a, p), bsm[o + p].w));
            });
            __syncthreads();
            float *t = a;
            a = b;
            b = t;
        }
        if (a != Z + o) {
            each(L, [&](int, int, int, int p) { Z[o + p] = a[p]; });
            __syncthreads();
        }
    }
    for (int l = le - 2; l >= lb; --l) {
        const Lev &L = e.lev[l], &C = e.lev[l + 1];
        const int oc = o;
        o -= L.sxy * L.nz;
        each(L, [&](int i, int j, int k, int p) {
            float acc = 0.f;
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float *x = Z + oc + ((k + c) >> 1) * C.sxy + ((j + b) >> 1) * C.sx;
                    acc += x[i >> 1] + x[(i + 1) >> 1];
                }
            R[o + p] = OMEGA * S[o + p] + 0.125f * acc;
        });
        __syncthreads();
        each(L, [&](int, int, int, int p) {
            Z[o + p] = (1.f - OMEGA) * R[o + p] +
                       OMEGA * (S[o + p] + __fdividef(faces(bsm + o, L, R + o, p), bsm[o + p].w));
        });
        __syncthreads();
    }
    const Lev &L = e.lev[lb];
    each(L, [&](int, int, int, int p) { L.z[p] = Z[p]; });
}

// Edge weights and ionic term (kept in z while the hierarchy is built) of a
// coarse level: from the FP64 weights and the code bytes of level 0, or
// from a coarse level.
template <bool FINE>
__global__ void k_mg_coarsen(mg::Lev F, mg::Lev C, const double *__restrict__ Wx, const double *__restrict__ Wy,
                             const double *__restrict__ Wz, const uint8_t *__restrict__ code, float kap0) {
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t >= C.nx * C.ny * C.nz) return;
    const int I = t % C.nx, J = (t / C.nx) % C.ny, K = t / (C.nx * C.ny);
    const int n[3] = {F.nx, F.ny, F.nz}, c[3] = {I, J, K};
    auto weight = [&](int d, const int (&x)[3]) -> float {
        if (FINE) {
            const double *W = d == 0 ? Wx : (d == 1 ? Wy : Wz);
            return (float)W[((long long)x[2] * F.ny + x[1]) * F.nx + x[0]];
        }
        const float4 q = F.cf[x[2] * F.sxy + x[1] * F.sx + x[0]];
        return d == 0 ? q.x : (d == 1 ? q.y : q.z);
    };
    float W[3];
    for (int d = 0; d < 3; ++d) {
        const int u = (d + 1) % 3, v = (d + 2) % 3;
        float sum = 0.f;
        for (int b = -1; b <= 1; ++b)
            for (int a = -1; a <= 1; ++a) {
                int x[3];
                x[u] = min(max(2 * c[u] + a, 0), n[u] - 1);
                x[v] = min(max(2 * c[v] + b, 0), n[v] - 1);
                x[d] = min(2 * c[d], n[d] - 2);
                const float p = weight(d, x);
                float w;
                if (2 * c[d] + 1 <= n[d] - 2) {
                    x[d] += 1;
                    const float q = weight(d, x);
                    w = 0.5f * (p * q / (p + q) + 0.25f * (p + q));
                } else {
                    w = p;  // one fine edge to the boundary
                }
                sum += (a ? 0.5f : 1.f) * (b ? 0.5f : 1.f) * w;
            }
        W[d] = c[d] < (d == 0 ? C.nx : (d == 1 ? C.ny : C.nz)) - 1 ? sum : 0.f;
    }
    float kap = 0.f;
    for (int e = 0; e < 27; ++e) {
        const int a = e % 3 - 1, b = (e / 3) % 3 - 1, g = e / 9 - 1;
        const int x = min(max(2 * I + a, 0), F.nx - 1), y = min(max(2 * J + b, 0), F.ny - 1),
                  z = min(max(2 * K + g, 0), F.nz - 1);
        const int p = z * F.sxy + y * F.sx + x;
        const float k = FINE ? ((code[p] & 1) ? 0.f : kap0) : F.z[p];
        kap += (a ? 0.5f : 1.f) * (b ? 0.5f : 1.f) * (g ? 0.5f : 1.f) * k;
    }
    const int p = K * C.sxy + J * C.sx + I;
    C.cf[p] = make_float4(W[0], W[1], W[2], 1.f);
    C.z[p] = kap;
}

__global__ void k_mg_diag(mg::Lev C) {
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t >= C.nx * C.ny * C.nz) return;
    const int I = t % C.nx, J = (t / C.nx) % C.ny, K = t / (C.nx * C.ny);
    if (!mg::interior(C, I, J, K)) return;
    const int p = K * C.sxy + J * C.sx + I;
    const float4 q = C.cf[p];
    C.cf[p].w = q.x + C.cf[p - 1].x + q.y + C.cf[p - C.sx].y + q.z + C.cf[p - C.sxy].z + C.z[p];
}

// ------------------------------------------------------------------- host --
struct MgState {
    mg::Entry e{};
    mg::Head *head = nullptr;    // device, of one-system launches
    float *v = nullptr;          // preconditioned residual (padded, level 0)
    void *mem = nullptr;         // coarse levels
    float *partials = nullptr;
};

// The levels of a grid; false when the hierarchy does not reach the bottom
// kernel's size (grids thinner than 9 nodes, or very long and thin ones):
// those keep the Jacobi preconditioner.
bool mg_levels(const PadGeo &g, mg::Entry &e) {
    using namespace mg;
    if (std::min(g.nx, std::min(g.ny, g.nz)) < 9) return false;
    int n[3] = {g.nx, g.ny, g.nz}, nl = 0;
    for (;; ++nl) {
        if (nl == LMAX) return false;
        Lev &L = e.lev[nl];
        L = Lev{};
        L.nx = n[0];
        L.ny = n[1];
        L.nz = n[2];
        L.sx = nl == 0 ? g.sx : ((n[0] + 3) & ~3);
        L.sxy = L.sx * n[1];
        if (std::min(n[0], std::min(n[1], n[2])) < 5) break;
        for (int d = 0; d < 3; ++d) n[d] = n[d] / 2 + 1;
    }
    e.nlev = nl + 1;
    long long nodes = 0;
    int b = e.nlev;
    while (b > 1) {
        const Lev &L = e.lev[b - 1];
        if (nodes + (long long)L.sxy * L.nz > BOT_NODES) break;
        nodes += (long long)L.sxy * L.nz;
        --b;
    }
    if (b == e.nlev) return false;
    e.nbot = b;
    // planes per work item: up to 8 coarse (16 fine) planes, fewer where that
    // leaves less than about four items an SM
    for (int l = 0; l < e.nbot; ++l) {
        const Lev &F = e.lev[l], &C = e.lev[l + 1];
        const long long cd = (long long)cdiv(C.nx - 1, CX) * cdiv(C.ny - 1, CY) * (C.nz - 2);
        const long long cu = (long long)cdiv(F.nx - 1, FX) * cdiv(F.ny - 1, FY) * (F.nz - 2);
        e.dk[l] = (int)std::max(1ll, std::min(8ll, cd / 608));
        e.uk[l] = (int)std::max(1ll, std::min(16ll, cu / 608));
    }
    return true;
}

void free_mg_state(pb_system *sys) {
    MgState *m = (MgState *)sys->mg;
    if (!m) return;
    dfree(m->head, sys->stream);
    dfree(m->v, sys->stream);
    dfree(m->mem, sys->stream);
    dfree(m->partials, sys->stream);
    delete m;
    sys->mg = nullptr;
}

size_t mg_bottom_bytes(const mg::Entry &e) {
    size_t n = 0;
    for (int l = e.nbot; l < e.nlev; ++l) n += (size_t)e.lev[l].sxy * e.lev[l].nz;
    return 28 * n;
}

pb_status mg_prepare() {
    static bool done = false;
    if (done) return PB_OK;
    const int most = 28 * mg::BOT_NODES;
    PB_CUDA_TRY(cudaFuncSetAttribute(k_mg_bottom<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    PB_CUDA_TRY(cudaFuncSetAttribute(k_mg_bottom<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    done = true;
    return PB_OK;
}

// hierarchy of a uniform system, built with its first mixed-precision solve
// (coefficients and grids do not change after that); sys->mg stays null on
// grids without one
pb_status build_mg_state(pb_system *sys, cudaStream_t s) {
    using namespace mg;
    if (sys->mg) return PB_OK;
    Entry e{};
    if (!mg_levels(sys->pad, e)) return PB_OK;
    pb_status rc = mg_prepare();
    if (rc != PB_OK) return rc;
    MgState *m = new (std::nothrow) MgState();
    if (!m) return PB_ERR_OOM;
    sys->mg = m;
    size_t bytes = 0;
    for (int l = 1; l < e.nlev; ++l) bytes += (size_t)e.lev[l].sxy * e.lev[l].nz * (sizeof(float4) + 8);
    e.nu0 = uitems(e, 0);
    m->head = (Head *)dalloc(sizeof(Head), s);
    m->v = (float *)dalloc(sizeof(float) * (size_t)sys->pad.Np, s);
    m->mem = dalloc(bytes, s);
    m->partials = (float *)dalloc(sizeof(float) * e.nu0, s);
    if (!m->head || !m->v || !m->mem || !m->partials) {
        free_mg_state(sys);
        return PB_ERR_OOM;
    }
    PB_CUDA_TRY(cudaMemsetAsync(m->head, 0, sizeof(Head), s));
    PB_CUDA_TRY(cudaMemsetAsync(m->v, 0, sizeof(float) * (size_t)sys->pad.Np, s));
    PB_CUDA_TRY(cudaMemsetAsync(m->mem, 0, bytes, s));
    e.lev[0].s = sys->z32;
    e.lev[0].z = m->v;
    char *at = (char *)m->mem;
    for (int l = 1; l < e.nlev; ++l) {
        Lev &L = e.lev[l];
        const size_t n = (size_t)L.sxy * L.nz;
        L.cf = (float4 *)at;
        L.s = (float *)(at + n * sizeof(float4));
        L.z = L.s + n;
        at += n * (sizeof(float4) + 8);
    }
    e.st = sys->st;
    e.code = sys->code;
    e.cp = make_c32(sys);
    e.partials = m->partials;
    for (int l = 1; l < e.nlev; ++l) {
        const Lev &F = e.lev[l - 1], &C = e.lev[l];
        const unsigned blocks = cdiv((long long)C.nx * C.ny * C.nz, 256);
        if (l == 1)
            k_mg_coarsen<true><<<blocks, 256, 0, s>>>(F, C, sys->W[0], sys->W[1], sys->W[2], sys->code, e.cp.kap);
        else
            k_mg_coarsen<false><<<blocks, 256, 0, s>>>(F, C, nullptr, nullptr, nullptr, nullptr, 0.f);
        k_mg_diag<<<blocks, 256, 0, s>>>(C);
        note_launch(1);
        PB_LAUNCH_CHECK();
    }
    for (int l = 1; l < e.nlev; ++l)  // z held the ionic terms
        PB_CUDA_TRY(cudaMemsetAsync(e.lev[l].z, 0, sizeof(float) * (size_t)e.lev[l].sxy * e.lev[l].nz, s));
    m->e = e;
    return PB_OK;
}

template <class K>
unsigned mg_resident(K kernel) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, mg::NT, 0) != cudaSuccess || per_sm <= 0) {
        cudaGetLastError();
        per_sm = 2;
    }
    return (unsigned)(per_sm * num_sms());
}

template <class... P, class... A>
void mg_launch(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, bool overlap,
               A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = overlap ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

// one V-cycle of one system (z32 -> v); returns the number of launches
int launch_vcycle(const pb_system *sys, cudaStream_t s) {
    using namespace mg;
    const MgState *m = (const MgState *)sys->mg;
    const Entry &e = m->e;
    static const unsigned rd0 = mg_resident(k_mg_down<true, true>), rd1 = mg_resident(k_mg_down<false, true>),
                          ru0 = mg_resident(k_mg_up<true, true>), ru1 = mg_resident(k_mg_up<false, true>);
    const Entry *none = nullptr;
    for (int l = 0; l < e.nbot; ++l) {
        const int n = ditems(e, l);
        if (l == 0)
            mg_launch(k_mg_down<true, true>, std::min<unsigned>(n, rd0), NT, 0, s, true, none, (const Head *)m->head, l,
                      n, e);
        else
            mg_launch(k_mg_down<false, true>, std::min<unsigned>(n, rd1), NT, 0, s, true, none, (const Head *)m->head,
                      l, n, e);
    }
    mg_launch(k_mg_bottom<true>, 1, BOT_T, mg_bottom_bytes(e), s, true, none, (const Head *)m->head, e);
    for (int l = e.nbot - 1; l >= 0; --l) {
        const int n = uitems(e, l);
        if (l == 0)
            mg_launch(k_mg_up<true, true>, std::min<unsigned>(n, ru0), NT, 0, s, true, none, m->head, l, n, e);
        else
            mg_launch(k_mg_up<false, true>, std::min<unsigned>(n, ru1), NT, 0, s, true, none, m->head, l, n, e);
    }
    return 2 * e.nbot + 1;
}
