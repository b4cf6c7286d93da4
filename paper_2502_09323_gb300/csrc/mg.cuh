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
// coarse levels stored weights and diagonals.  The levels
// whose data fits one block's shared memory are solved by one block per
// system in one launch (k_mg_bottom).  The up kernel of level 0 also sums
// rho = r.z and takes the CG step beta = rho / rho_old.
//
// Measured (GB300, solves to 1e-12): 257^3 155.6 -> 13.1 ms (1,127 -> 30
// iterations; 33 to 36 are launched, as the host looks every other one), 65^3
// 30.1 -> 2.1 ms, a batch of 24 systems of 97^3 to 161^3 229 -> 51 ms.
//
// Bounds: down reads s and a code byte per fine node and writes an eighth of
// a value; up reads s, an eighth of a value and a code byte and writes z.
#pragma once

namespace mg {

constexpr int LMAX = 12;            // levels at most
constexpr float OMEGA = 0.85f;      // Jacobi damping (0.8 to 0.9 take the same iterations)
constexpr int BOT_T = 1024;         // threads of the bottom kernel
// shared memory of a node of the bottom kernel: the blob's four coefficients
// and three lists, and three vectors; nodes of all its levels at most
template <typename T>
constexpr int BLOB_BYTES = 4 * sizeof(T) + 6;
template <typename T>
constexpr int BOT_BYTES = 7 * sizeof(T) + 6;
template <typename T>
constexpr int BOT_NODES = sizeof(T) == 4 ? 6600 : 3600;
constexpr int SWEEPS = 8;           // Jacobi sweeps on the coarsest level
// Tiles of the coarse levels.  Down: 32 x 6 coarse nodes from node (1 + 32 bx, 1 + 6 by), whose
// residuals are 13 rows of 17 units of 4 fine nodes; the first and the last
// unit of a row need no neighbour outside it.  221 threads take a unit each,
// 34 more the halo rows.  Up: 64 x 16 fine nodes from (64 bx, 1 + 16 by), 16
// units a row, and a halo row on either side: 288 threads.
constexpr int CX = 32, CY = 6, DU = 17, DR = 2 * CY + 1, DNT = 256;
constexpr int FX = 64, FY = 16, UU = 16, UNT = 16 * (FY + 2);
constexpr int RG = 4;               // planes of one partial of rho

template <typename T>
struct LevT {
    int nx, ny, nz, sx, sxy;    // sx a multiple of 4 above the bottom kernel's levels, nx there
    T *s, *z;                   // D^-1 b, solution (level 0: the solver's s and v)
    T *wx, *wy, *wz, *dg;       // weights of the +x, +y, +z edges, diagonal (levels >= 1)
    T *di, *r;                  // FP64 cycle: 1 / diagonal, work vector
};
using Lev = LevT<float>;

// One system (device memory, or the kernel parameter of a one-system launch)
struct Entry {
    using T = float;
    Lev lev[LMAX];
    int nlev, nbot;                 // levels; first level of the bottom kernel
    int dbase[LMAX], ubase[LMAX];   // first work item of this system in a level's launches
    int dk[LMAX], uk[LMAX];         // planes per work item (coarse planes down, fine planes up)
    CgState *st;
    const uint8_t *code;
    CoefC32 cp;
    float dg_in, dg_out;            // diagonals of the two pure media
    float *partials;                // rho of every RG planes of each tile of level 0
    int nu0;                        // their number
    void *blob;                     // of the bottom kernel (k_mg_pack)
    int bot;                        // its nodes, rounded up to a multiple of 8
    CUtensorMap sd, cd, su, cu;     // s and codes of level 0: boxes of k_mg_down0, of k_mg_up0
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
    const int cy = l == 0 && e.code ? 8 : CY;  // k_mg_down0's tile
    return ((c.nx - 2 + CX - 1) / CX) * ((c.ny - 2 + cy - 1) / cy) * ((c.nz - 2 + e.dk[l] - 1) / e.dk[l]);
}
__host__ __device__ inline int uitems(const Entry &e, int l) {
    if (l >= e.nbot) return 0;
    const Lev &f = e.lev[l];
    return ((f.nx - 1 + FX - 1) / FX) * ((f.ny - 2 + FY - 1) / FY) * ((f.nz - 2 + e.uk[l] - 1) / e.uk[l]);
}

__device__ __forceinline__ float quotient(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double quotient(double a, double b) { return a * rcp_fp64(b); }  // b a diagonal

__device__ __forceinline__ float4 f4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 ldg4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }

// Operator data of a unit (4 nodes of a row) in one plane.  Level 0: its code
// bytes, those of the row below and of the node to the left.  Coarse levels:
// the weights and the diagonal.
struct Codes {
    uint32_t c = 0, cy = 0, cl = 0;
};
struct Weights {
    float4 x = {}, y = {}, z = {}, ym = {}, d = {1.f, 1.f, 1.f, 1.f};
    float xl = 0.f;
    __device__ __forceinline__ void load(const Entry &, const Lev &L, int p) {
        x = f4(L.wx + p);
        y = f4(L.wy + p);
        z = f4(L.wz + p);
        ym = f4(L.wy + p - L.sx);
        d = f4(L.dg + p);
        xl = L.wx[p - 1];
    }
};

// sum over the six faces of W times the neighbour, and the diagonal, of the
// nodes of a unit; l, r: neighbours in x.  Level 0, a unit with listed edges:
// below holds its codes in plane k - 1.  The weights' arrays are dense, so the
// whole unit's are loaded in six independent loads and the unlisted ones are
// passed over: a load under a condition of its own for each face waited for
// the one before it (about 10,000 cycles a plane for the slowest warp).
__device__ __forceinline__ void listed_sums(const CoefC32 &cp, const Lev &L, int p, const Codes &o, uint32_t below,
                                            const float4 &x, float l, float r, const float4 &ym, const float4 &yp,
                                            const float4 &zm, const float4 &zp, float (&sum)[4], float (&d)[4]) {
    const float4 g1 = ldg4(cp.wx + p), g2 = ldg4(cp.wy + p - L.sx), g3 = ldg4(cp.wy + p),
                 g4 = ldg4(cp.wz + p - L.sxy), g5 = ldg4(cp.wz + p);
    const float g0 = __ldg(cp.wx + p - 1);
    const float xx[6] = {l, x.x, x.y, x.z, x.w, r};
    const float my[4] = {ym.x, ym.y, ym.z, ym.w}, py[4] = {yp.x, yp.y, yp.z, yp.w};
    const float mz[4] = {zm.x, zm.y, zm.z, zm.w}, pz[4] = {zp.x, zp.y, zp.z, zp.w};
    const float v1[4] = {g1.x, g1.y, g1.z, g1.w}, v2[4] = {g2.x, g2.y, g2.z, g2.w}, v3[4] = {g3.x, g3.y, g3.z, g3.w};
    const float v4[4] = {g4.x, g4.y, g4.z, g4.w}, v5[4] = {g5.x, g5.y, g5.z, g5.w};
    float wl = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t c = o.c >> (8 * q);
        const float w = (c & 1u) ? cp.w_in : cp.w_out;
        if (q == 0) wl = (o.cl & 2u) ? g0 : w;
        else wl = ((o.c >> (8 * q - 8)) & 2u) ? wl : w;
        const float w1 = (c & 2u) ? v1[q] : w;
        const float w2 = ((o.cy >> (8 * q)) & 4u) ? v2[q] : w;
        const float w3 = (c & 4u) ? v3[q] : w;
        const float w4 = ((below >> (8 * q)) & 8u) ? v4[q] : w;
        const float w5 = (c & 8u) ? v5[q] : w;
        d[q] = (((((wl + w1) + w2) + w3) + w4) + w5) + ((c & 1u) ? 0.f : cp.kap);
        sum[q] = ((wl * xx[q] + w1 * xx[q + 2]) + (w2 * my[q] + w3 * py[q])) + (w4 * mz[q] + w5 * pz[q]);
        wl = w1;
    }
}
__device__ __forceinline__ void face_sums(const Entry &, const Lev &, int, const Weights &o, const Weights &b,
                                          const float4 &x, float l, float r, const float4 &ym, const float4 &yp,
                                          const float4 &zm, const float4 &zp, float (&sum)[4], float (&d)[4]) {
    sum[0] = ((o.xl * l + o.x.x * x.y) + (o.ym.x * ym.x + o.y.x * yp.x)) + (b.z.x * zm.x + o.z.x * zp.x);
    sum[1] = ((o.x.x * x.x + o.x.y * x.z) + (o.ym.y * ym.y + o.y.y * yp.y)) + (b.z.y * zm.y + o.z.y * zp.y);
    sum[2] = ((o.x.y * x.y + o.x.z * x.w) + (o.ym.z * ym.z + o.y.z * yp.z)) + (b.z.z * zm.z + o.z.z * zp.z);
    sum[3] = ((o.x.z * x.z + o.x.w * r) + (o.ym.w * ym.w + o.y.w * yp.w)) + (b.z.w * zm.w + o.z.w * zp.w);
    d[0] = o.d.x;
    d[1] = o.d.y;
    d[2] = o.d.z;
    d[3] = o.d.w;
}

template <typename T>
__device__ __forceinline__ bool interior(const LevT<T> &L, int i, int j, int k) {
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

// Residual after the pre-smoothing step and its restriction, on coarse levels
// (and a lattice's level 0).  A block marches
// over the coarse planes of its tile: a thread keeps its unit's s of three
// planes in registers, rows are exchanged through shared memory (three planes
// of s, two of the residual, so that one barrier a fine plane suffices), and a
// plane's loads are issued one plane ahead.
template <bool SINGLE>
__global__ void __launch_bounds__(mg::DNT, 3)
k_mg_down(const mg::Entry *__restrict__ tab, const mg::Head *__restrict__ head, int l, int total,
          const __grid_constant__ mg::Entry e0) {
    using namespace mg;
    __shared__ __align__(16) float sp[3][DR + 2][4 * DU];
    __shared__ __align__(16) float rb[2][DR][4 * DU];
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    // unit u of row r of the tile's fine rows - 1 .. DR (rows - 1 and DR: halo)
    const bool halo = tid >= DR * DU;
    const int h = tid - DR * DU;
    const int u = halo ? h % DU : tid % DU, r = halo ? (h < DU ? -1 : DR) : tid / DU;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int nsys = SINGLE ? 1 : head->nsys;
    if (!SINGLE) total = head->dtotal[l];
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        const Entry &e = SINGLE ? e0 : tab[find_sys(tab, nsys, it, &Entry::dbase, l)];
        if (*(volatile int *)&e.st->done) continue;
        const Lev L = e.lev[l], C = e.lev[l + 1];
        const int li = SINGLE ? it : it - e.dbase[l];
        const int xt = (C.nx - 2 + CX - 1) / CX, yt = (C.ny - 2 + CY - 1) / CY;
        const int col = li % (xt * yt), ch = li / (xt * yt);
        const int I0 = 1 + (col % xt) * CX, J0 = 1 + (col / xt) * CY;
        const int K0 = 1 + ch * e.dk[l], K1 = min(K0 + e.dk[l], C.nz - 1);
        const int ka = 2 * K0 - 1, kb = 2 * K1 - 1;  // fine planes ka .. kb of the residual
        const int ib = 2 * I0 - 2 + 4 * u, j = 2 * J0 - 1 + r;
        const bool there = h < 2 * DU && ib < L.sx && j >= 0 && j < L.ny;
        const bool row = there && !halo && j <= L.ny - 2;  // j >= 1
        const int pj = j * L.sx + ib;
        auto load = [&](int k) {
            return there && k < L.nz ? f4(L.s + (k * L.sxy + pj)) : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        float4 sm, sc, sn, s2;
        Weights ob, oc, on;
        sm = halo ? make_float4(0.f, 0.f, 0.f, 0.f) : load(ka - 1);
        sc = load(ka);
        sn = load(ka + 1);
        if (row) {
            ob.load(e, L, (ka - 1) * L.sxy + pj);
            oc.load(e, L, ka * L.sxy + pj);
        }
        __syncthreads();  // the previous item's last reads
        if (h < 2 * DU) *reinterpret_cast<float4 *>(&sp[ka % 3][r + 1][4 * u]) = sc;
        float acc = 0.f;
        for (int k = ka; k <= kb + 1; ++k) {
            if (k < kb && h < 2 * DU) *reinterpret_cast<float4 *>(&sp[(k + 1) % 3][r + 1][4 * u]) = sn;
            __syncthreads();
            if (k < kb) {
                s2 = load(k + 2);
                if (row) on.load(e, L, (k + 1) * L.sxy + pj);
            }
            if (k <= kb && !halo) {
                float v[4] = {0.f, 0.f, 0.f, 0.f};
                if (row && k <= L.nz - 2) {
                    const float (*s)[4 * DU] = sp[k % 3];
                    const float xl = u > 0 ? s[r + 1][4 * u - 1] : 0.f, xr = u < DU - 1 ? s[r + 1][4 * u + 4] : 0.f;
                    float sum[4], d[4];
                    face_sums(e, L, k * L.sxy + pj, oc, ob, sc, xl, xr, f4(&s[r][4 * u]), f4(&s[r + 2][4 * u]), sm, sn,
                              sum, d);
                    const float s4[4] = {sc.x, sc.y, sc.z, sc.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (ib + q >= 1 && ib + q <= L.nx - 2) v[q] = (1.f - OMEGA) * d[q] * s4[q] + OMEGA * sum[q];
                }
                *reinterpret_cast<float4 *>(&rb[k & 1][r][4 * u]) = make_float4(v[0], v[1], v[2], v[3]);
            }
            if (k > ka && ty < CY) {  // restrict plane k - 1
                float t = 0.f;
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const float *x = &rb[(k - 1) & 1][2 * ty + b][2 * tx + 1];
                    const float v = x[1] + 0.5f * (x[0] + x[2]);
                    t += b == 1 ? v : 0.5f * v;
                }
                if ((k - 1) & 1) {
                    acc += 0.5f * t;
                    const int K = (k - 2) >> 1, I = I0 + tx, J = J0 + ty;
                    if (k - 1 > ka && I <= C.nx - 2 && J <= C.ny - 2) {
                        const int pc = K * C.sxy + J * C.sx + I;
                        C.s[pc] = __fdividef(acc, __ldg(C.dg + pc));
                    }
                    acc = 0.5f * t;
                } else {
                    acc += t;
                }
            }
            sm = sc;
            sc = sn;
            sn = s2;
            ob = oc;
            oc = on;
        }
    }
}

// Interpolated correction and post-smoothing step of a coarse level.  A
// block marches over the fine planes of its tile: a thread keeps its unit's v
// of three planes and the coarse correction, interpolated in y, of two coarse
// planes in registers; rows of v are exchanged through three planes of shared
// memory (one barrier a plane).
template <bool SINGLE>
__global__ void __launch_bounds__(mg::UNT, 2)
k_mg_up(const mg::Entry *__restrict__ tab, const mg::Head *__restrict__ head, int l, int total,
        const __grid_constant__ mg::Entry e0) {
    using namespace mg;
    constexpr int VW = FX + 8;  // a row: col - 1 at [3], cols 0 .. 63 from [4], col 64 at [68]
    __shared__ __align__(16) float vp[3][FY + 2][VW];
    const int tid = threadIdx.x;
    const int u = tid & 15, r = tid >> 4;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int nsys = SINGLE ? 1 : head->nsys;
    if (!SINGLE) total = head->utotal[l];
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        const Entry &e = SINGLE ? e0 : tab[find_sys(tab, nsys, it, &Entry::ubase, l)];
        if (*(volatile int *)&e.st->done) continue;
        const Lev L = e.lev[l], C = e.lev[l + 1];
        const int li = SINGLE ? it : it - e.ubase[l];
        const int xt = (L.nx - 1 + FX - 1) / FX, yt = (L.ny - 2 + FY - 1) / FY;
        const int col = li % (xt * yt), ch = li / (xt * yt);
        const int i0 = (col % xt) * FX, ib = i0 + 4 * u, j = (col / xt) * FY + r;
        const int k0 = 1 + ch * e.uk[l], k1 = min(k0 + e.uk[l], L.nz - 1);
        const bool row = ib <= L.nx - 2 && j >= 1 && j <= L.ny - 2;
        const bool own = row && r >= 1 && r <= FY;
        const int pj = j * L.sx + ib;
        const bool left = u == 0 && i0 > 0 && row, right = u == UU - 1 && ib + 4 <= L.nx - 2 && row;
        // s of a unit, and of the columns beside the tile
        struct S {
            float4 s;
            float x;
        };
        auto load_s = [&](int k) {
            S t = {make_float4(0.f, 0.f, 0.f, 0.f), 0.f};
            if (row && k >= 1 && k <= L.nz - 2) {
                const float *p = L.s + (k * L.sxy + pj);
                t.s = f4(p);
                if (left) t.x = p[-1];
                if (right) t.x = p[4];
            }
            return t;
        };
        // coarse correction at columns ib/2 .. ib/2 + 2 (and ib/2 - 1 beside
        // the tile), interpolated to row j, of coarse plane K
        struct E {
            float x, y, z, l;
        };
        const int I = ib >> 1, pa = (j >> 1) * C.sx + I, pb = ((j + 1) >> 1) * C.sx + I;
        const bool third = I + 2 < C.sx;
        auto load_e = [&](int K) {
            E t = {0.f, 0.f, 0.f, 0.f};
            if (row && K < C.nz) {
                const float *a = C.z + (K * C.sxy + pa), *b = C.z + (K * C.sxy + pb);
                t.x = 0.5f * (a[0] + b[0]);
                t.y = 0.5f * (a[1] + b[1]);
                if (third) t.z = 0.5f * (a[2] + b[2]);
                if (left) t.l = 0.5f * (a[-1] + b[-1]);
            }
            return t;
        };
        // v = w s + P e of plane k, from the coarse planes k/2 and (k+1)/2;
        // zero off the interior
        auto make_v = [&](int k, const S &s, const E &a, const E &b) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row && k >= 1 && k <= L.nz - 2) {
                const float x = 0.5f * (a.x + b.x), y = 0.5f * (a.y + b.y), z = 0.5f * (a.z + b.z);
                if (ib >= 1) v.x = OMEGA * s.s.x + x;
                if (ib + 1 <= L.nx - 2) v.y = OMEGA * s.s.y + 0.5f * (x + y);
                if (ib + 2 <= L.nx - 2) v.z = OMEGA * s.s.z + y;
                if (ib + 3 <= L.nx - 2) v.w = OMEGA * s.s.w + 0.5f * (y + z);
                float *out = vp[k % 3][r];
                if (left) out[3] = OMEGA * s.x + 0.5f * (0.5f * (a.l + b.l) + x);
                if (right) out[4 + FX] = OMEGA * s.x + z;
            }
            *reinterpret_cast<float4 *>(&vp[k % 3][r][4 + 4 * u]) = v;
            return v;
        };
        S sa = load_s(k0 - 1), sc = load_s(k0), sn = load_s(k0 + 1);
        E ea = load_e((k0 - 1) >> 1), eb = load_e(k0 >> 1), ec = load_e((k0 + 1) >> 1), en = load_e((k0 + 2) >> 1);
        Weights ob, oc, on;
        if (own) {
            ob.load(e, L, (k0 - 1) * L.sxy + pj);
            oc.load(e, L, k0 * L.sxy + pj);
        }
        __syncthreads();  // the previous item's last reads
        if (u == 0 && !left)
            for (int q = 0; q < 3; ++q) vp[q][r][3] = 0.f;
        if (u == UU - 1 && !right)
            for (int q = 0; q < 3; ++q) vp[q][r][4 + FX] = 0.f;
        float4 vm = make_v(k0 - 1, sa, ea, eb);
        float4 vc = make_v(k0, sc, eb, ec);
        // coarse planes of v(k + 1): (k + 1) / 2 and (k + 2) / 2
        ea = ec;
        eb = en;
        for (int k = k0; k < k1; ++k) {
            const float4 vn = make_v(k + 1, sn, ea, eb);
            __syncthreads();
            // issue the next plane's loads
            S s2 = load_s(k + 2);
            ec = eb;
            if (!((k + 1) & 1)) ec = load_e((k + 3) >> 1);
            if (own) {
                if (k + 1 < k1) on.load(e, L, (k + 1) * L.sxy + pj);
                const float (*v)[VW] = vp[k % 3];
                float sum[4], d[4];
                face_sums(e, L, k * L.sxy + pj, oc, ob, vc, v[r][3 + 4 * u], v[r][8 + 4 * u], f4(&v[r - 1][4 + 4 * u]),
                          f4(&v[r + 1][4 + 4 * u]), vm, vn, sum, d);
                const float v4[4] = {vc.x, vc.y, vc.z, vc.w}, s4[4] = {sc.s.x, sc.s.y, sc.s.z, sc.s.w};
                float z[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    z[q] = (1.f - OMEGA) * v4[q] + OMEGA * (s4[q] + __fdividef(sum[q], d[q]));
                    if (ib + q < 1 || ib + q > L.nx - 2) z[q] = 0.f;
                }
                *reinterpret_cast<float4 *>(L.z + (k * L.sxy + pj)) = make_float4(z[0], z[1], z[2], z[3]);
            }
            vm = vc;
            vc = vn;
            sc = sn;
            sn = s2;
            ea = ((k + 1) & 1) ? eb : ea;
            eb = ec;
            ob = oc;
            oc = on;
        }
    }
}

// ---- level 0 of a solver's grid: two rows a thread
// A thread takes a unit of four nodes in two neighbouring rows.  The planes of
// s and codes come in by TMA, NS in shared memory and up to three ahead of
// their use (the first thread issues them, out-of-range elements are zero);
// arithmetic is in packed FP32 pairs; weights of unlisted units come from a
// table by the units' four solute bits, those of listed ones from listed_sums.
//
// 257^3, down and up: one row a thread with loads into registers a plane
// ahead 102 and 139 us; this form 70 and 88 us by the same timing, 61 and 73 us
// among the other kernels of a solve (21 and 25 us at the measured copy rate,
// all that is read and written counted).  What was in the way, one after the other: a gather of its own for each listed face (below);
// parameters read again after every asm statement (hence the local copies);
// resident blocks that walked over their items, so that a block with the
// molecule's surface in both of its items held up the launch (a one-system
// launch now has a block an item); asynchronous copies of each thread's own,
// 60 instructions a plane (TMA); the listed weights' latency (prefetched a
// plane ahead).  Counters now (257^3): instructions issue in 44 and 47 % of
// the cycles, the DRAM moves at 25 % of its rate; the listed weights' loads
// (down) and the barrier of each plane (up) are what warps wait for most.
namespace mg {
constexpr int C0Y = 8, D0P = C0Y + 1, D0NT = 160;  // down: 32 x 8 coarse nodes, nine row pairs of 17 units
constexpr int U0NT = 192;                          // up: eight row pairs, a warp of halo rows, a warp of halo columns
constexpr int NS = 4;                              // planes of s and codes in shared memory
constexpr int D0R = 2 * D0P + 1, D0W = 4 * DU;     // the down kernel's box of s
constexpr int U0R = FY + 2, U0W = FX + 8;          // the up kernel's: columns from i0 - 4
constexpr int C0W = FX + 32;                       // codes: columns from 16 to the left
constexpr int up128(int b) { return (b + 127) & ~127; }
// The ring of planes of one block.  Planes are counted over the whole launch.
// Every wait is bounded by tma::g_slot_wait_limit, as in the stencil kernels.
// After one that gives up, the thread polls each slot once; the first thread,
// which issues the copies, first waits (with a limit of its own) for those in
// flight, and issues no more: it did not see their slots filled.  The block
// computes on with whatever its slots hold (no address depends on it) and says
// so in the solver's state (status 3, whose correction is dropped).
template <int R, int W, int RC>  // rows and columns of s, rows of codes
struct Ring {
    static constexpr int SB = up128(4 * R * W), CB = up128(RC * C0W);
    struct Mem {
        uint8_t s[NS][SB], c[NS][CB];
    };
    Mem &m;
    uint32_t bar;        // NS mbarriers
    int n = 0;           // planes waited for
    int who;             // the thread; another number for a first one that gave up
    bool bad = false;    // a wait gave up
    __device__ __forceinline__ Ring(Mem &mem, uint64_t *bars) : m(mem), bar(tma::smem_u32(bars)), who(threadIdx.x) {
        if (threadIdx.x == 0) {
            for (int q = 0; q < NS; ++q) tma::mbar_init(bar + 8 * q, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    }
    // plane k, the `at`-th after those waited for
    __device__ __forceinline__ void issue(const CUtensorMap &sm, const CUtensorMap &cm, int x, int y, int k, int at) {
        if (who == 0) {
            const int q = (n + at) & (NS - 1);
            const uint32_t b = bar + 8 * q;
            tma::mbar_expect_tx(b, 4 * R * W + RC * C0W);
            tma::tma_load3(tma::smem_u32(m.s[q]), &sm, x - (W == U0W ? 4 : 0), y, k, b);
            tma::tma_load3(tma::smem_u32(m.c[q]), &cm, x - 16, y, k, b);
        }
    }
    // gives up; `flying` planes from the next one on may be in flight
    __device__ __forceinline__ void give_up(int flying) {
        bad = true;
        if (who == 0)
            for (int q = n; q < n + flying; ++q)
                tma::mbar_wait(bar + 8 * (q & (NS - 1)), (q / NS) & 1, tma::TMA_WAIT_LIMIT);
        who = -1;
    }
    // for the next plane; `after` it are in flight
    __device__ __forceinline__ void wait(int after) {
        const uint32_t b = bar + 8 * (n & (NS - 1)), parity = (n / NS) & 1;
        if (!tma::mbar_try(b, parity) && !tma::mbar_wait(b, parity, bad ? 0 : tma::g_slot_wait_limit)) give_up(1 + after);
        ++n;
    }
    __device__ __forceinline__ const float (*s(int back) const)[W] {  // plane back before the last one waited for
        return reinterpret_cast<const float (*)[W]>(m.s[(n - 1 - back) & (NS - 1)]);
    }
    __device__ __forceinline__ const uint8_t (*c(int back) const)[C0W] {
        return reinterpret_cast<const uint8_t (*)[C0W]>(m.c[(n - 1 - back) & (NS - 1)]);
    }
    __device__ __forceinline__ static void fail(CgState *st) {
        if (st->done) return;
        st->status = 3;
        st->done = 1;
    }
    __device__ __forceinline__ void report(CgState *st) {
        if (bad) fail(st);
    }
};
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool there) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tma::smem_u32(dst)), "l"(src), "r"(there ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src, bool there) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tma::smem_u32(dst)), "l"(src), "r"(there ? 4 : 0)
                 : "memory");
}
struct Pair4 {  // four values as two packed pairs
    float2 a, b;
};
__device__ __forceinline__ Pair4 p4(const float4 &v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 f4(const Pair4 &v) { return make_float4(v.a.x, v.a.y, v.b.x, v.b.y); }
__device__ __forceinline__ Pair4 operator+(const Pair4 &x, const Pair4 &y) {
    return {__fadd2_rn(x.a, y.a), __fadd2_rn(x.b, y.b)};
}
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ Pair4 scale(float c, const Pair4 &x) {
    return {__fmul2_rn(both(c), x.a), __fmul2_rn(both(c), x.b)};
}
__device__ __forceinline__ Pair4 fma4(float c, const Pair4 &x, const Pair4 &y) {  // c x + y
    return {__ffma2_rn(both(c), x.a, y.a), __ffma2_rn(both(c), x.b, y.b)};
}
__device__ __forceinline__ Pair4 fma4(const Pair4 &c, const Pair4 &x, const Pair4 &y) {
    return {__ffma2_rn(c.a, x.a, y.a), __ffma2_rn(c.b, x.b, y.b)};
}
__device__ __forceinline__ Pair4 mul4(const Pair4 &x, const Pair4 &y) {
    return {__fmul2_rn(x.a, y.a), __fmul2_rn(x.b, y.b)};
}
// the six neighbours of a unit's nodes added up
__device__ __forceinline__ Pair4 neighbours(const Pair4 &c, float l, float r, const Pair4 &ym, const Pair4 &yp,
                                            const Pair4 &zm, const Pair4 &zp) {
    const float2 mid = make_float2(c.a.y, c.b.x);
    const Pair4 x = {__fadd2_rn(make_float2(l, c.a.x), mid), __fadd2_rn(mid, make_float2(c.b.y, r))};
    return x + (ym + yp) + (zm + zp);
}
// byte offset into a table of 16 float4: the solute bits of four codes
__device__ __forceinline__ uint32_t media(uint32_t c) { return ((c & 0x01010101u) * 0x01020408u) >> 20; }
__device__ __forceinline__ Pair4 entry(const float4 *table, uint32_t at) {
    return p4(*reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(table) + at));
}
// fills entry t of a table with one of two values by each bit of t
__device__ __forceinline__ void fill_media(float4 *table, int t, float in, float out) {
    table[t] = make_float4((t & 1) ? in : out, (t & 2) ? in : out, (t & 4) ? in : out, (t & 8) ? in : out);
}
__device__ __forceinline__ bool listed(const Codes &o, uint32_t below) {
    const uint32_t cx = (o.c << 8) | o.cl;
    return ((o.c & 0x0E0E0E0Eu) | (cx & 0x02020202u) | (o.cy & 0x04040404u) | (below & 0x08080808u)) != 0u;
}
__device__ __forceinline__ void listed_sums(const CoefC32 &cp, const Lev &L, int p, const Codes &o, uint32_t below,
                                            const Pair4 &c, float l, float r, const Pair4 &ym, const Pair4 &yp,
                                            const Pair4 &zm, const Pair4 &zp, Pair4 &sum, Pair4 &d) {
    // the surface mostly goes on in the next plane
    tma::prefetch_l1(cp.wx + p + L.sxy);
    tma::prefetch_l1(cp.wy + p + L.sxy - L.sx);
    tma::prefetch_l1(cp.wy + p + L.sxy);
    tma::prefetch_l1(cp.wz + p + L.sxy);
    float s4[4], d4[4];
    listed_sums(cp, L, p, o, below, f4(c), l, r, f4(ym), f4(yp), f4(zm), f4(zp), s4, d4);
    sum = {make_float2(s4[0], s4[1]), make_float2(s4[2], s4[3])};
    d = {make_float2(d4[0], d4[1]), make_float2(d4[2], d4[3])};
}
}  // namespace mg

// Residual and restriction of level 0.  Row pair p of a tile is rows 2 J - 1
// and 2 J of its coarse row J; its share of the sums across y is formed in the
// thread, half of the next pair's first row and the last column of the unit
// to the left come through shared memory.  Planes are taken in pairs.
template <bool SINGLE>
__global__ void __launch_bounds__(mg::D0NT, 4)
k_mg_down0(const mg::Entry *__restrict__ tab, const mg::Head *__restrict__ head, int total,
           const __grid_constant__ mg::Entry e0) {
    using namespace mg;
    using R = Ring<D0R, D0W, D0R>;
    __shared__ __align__(128) R::Mem planes;
    __shared__ __align__(16) float half[2][D0P][D0W];  // half the residual of each pair's first row
    __shared__ float last[2][D0P][DU];                 // each unit's last column of a pair's share
    __shared__ float4 tw[16], td[16];                  // omega w and (1 - omega) d
    __shared__ uint64_t bars[NS];
    const int tid = threadIdx.x;
    const int pr = tid / DU, u = tid - pr * DU;  // pair and unit of a thread
    const bool work = pr < D0P;
    const int ra = work ? 2 * pr + 1 : 1, x = 4 * u;  // row of the box
    R ring(planes, bars);
    // a limit of no polls gives up before anything is issued: a wait looks at
    // its slot once before it counts
    const bool no_polls = tma::g_slot_wait_limit == 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int nsys = SINGLE ? 1 : head->nsys;
    if (!SINGLE) total = head->dtotal[0];
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        const Entry &e = SINGLE ? e0 : tab[find_sys(tab, nsys, it, &Entry::dbase, 0)];
        // one answer for the block; and the previous item's last reads, the barriers' initialisation
        if (__syncthreads_or(*(volatile int *)&e.st->done | (int)no_polls)) {
            if (no_polls) ring.fail(e.st);
            continue;
        }
        // local copies: the asm statements below would have e read again
        const Lev L = e.lev[0], C = e.lev[1];
        const CoefC32 cp = e.cp;
        const int li = SINGLE ? it : it - e.dbase[0];
        const int xt = (C.nx - 2 + CX - 1) / CX, yt = (C.ny - 2 + C0Y - 1) / C0Y;
        const int col = li % (xt * yt), ch = li / (xt * yt);
        const int I0 = 1 + (col % xt) * CX, J0 = 1 + (col / xt) * C0Y;
        const int K0 = 1 + ch * e.dk[0], K1 = min(K0 + e.dk[0], C.nz - 1);
        const int ka = 2 * K0 - 1, kb = 2 * K1 - 1;
        const int i0 = 2 * I0 - 2, jb = 2 * J0 - 2, ib = i0 + x, ja = jb + ra;
        const bool rowA = work && ib < L.sx && ja <= L.ny - 2, rowB = rowA && ja + 1 <= L.ny - 2 && pr < D0P - 1;
        const int pj = ja * L.sx + ib;
        const bool edge = ib < 1 || ib + 3 > L.nx - 2;
        auto clip = [&](Pair4 &v) {  // nodes of the unit that are no unknowns
            if (ib < 1 || ib > L.nx - 2) v.a.x = 0.f;
            if (ib + 1 > L.nx - 2) v.a.y = 0.f;
            if (ib + 2 > L.nx - 2) v.b.x = 0.f;
            if (ib + 3 > L.nx - 2) v.b.y = 0.f;
        };
        const int I = I0 - 1 + 2 * u, J = J0 + pr;  // the thread's coarse nodes
        const bool in0 = pr < C0Y && J <= C.ny - 2 && u > 0 && I <= C.nx - 2;
        const bool in1 = pr < C0Y && J <= C.ny - 2 && u < DU - 1 && I + 1 <= C.nx - 2;
        const int pcj = J * C.sx + I;
        const int first = min(4, kb - ka + 3);  // planes to begin with
        for (int q = 0; q < first; ++q) ring.issue(e.sd, e.cd, i0, jb, ka - 1 + q, q);
        if (tid < 16) fill_media(tw, tid, OMEGA * cp.w_in, OMEGA * cp.w_out);
        else if (tid < 32) fill_media(td, tid - 16, (1.f - OMEGA) * e.dg_in, (1.f - OMEGA) * e.dg_out);
        ring.wait(first - 1);
        ring.wait(first - 2);
        auto word = [&](const uint8_t (*c)[C0W], int r) { return *reinterpret_cast<const uint32_t *>(&c[r][16 + x]); };
        uint32_t bA = word(ring.c(1), ra), bB = word(ring.c(1), ra + 1);  // codes of plane k - 1
        Pair4 mA = p4(f4(&ring.s(1)[ra][x])), mB = p4(f4(&ring.s(1)[ra + 1][x]));
        Pair4 cA = p4(f4(&ring.s(0)[ra][x])), cB = p4(f4(&ring.s(0)[ra + 1][x])), share = {};
        float acc0 = 0.f, acc1 = 0.f, dc0 = 1.f, dc1 = 1.f;
        // plane k, an odd one or not, and the restriction of the one before
        auto step = [&](int k, auto odd, bool compute) {
            constexpr bool ODD = decltype(odd)::value;
            const bool done = !ODD && k - 1 > ka;  // completes coarse nodes
            const int pc = ((k - (ODD ? 1 : 2)) >> 1) * C.sxy + pcj;
            if (compute) ring.wait(k + 2 <= kb + 1);  // plane k + 1
            __syncthreads();
            if (ODD && k > ka) {  // their diagonals, a plane ahead
                if (in0) dc0 = __ldg(C.dg + pc);
                if (in1) dc1 = __ldg(C.dg + pc + 1);
            }
            Pair4 next = {};
            if (compute) {
                if (k + 3 <= kb + 1) ring.issue(e.sd, e.cd, i0, jb, k + 3, 1);  // over plane k - 1
                const float (*s)[D0W] = ring.s(1), (*sn)[D0W] = ring.s(0);
                const uint8_t (*cd)[C0W] = ring.c(1);
                const Pair4 nA = p4(f4(&sn[ra][x])), nB = p4(f4(&sn[ra + 1][x]));
                Pair4 rA = {}, rB = {};
                const uint32_t nbA = word(cd, ra), nbB = word(cd, ra + 1);
                if (rowA && k <= L.nz - 2) {
                    const int p = k * L.sxy + pj;
                    Codes o;
                    auto residual = [&](int q, int r, const Pair4 &c, const Pair4 &ym, const Pair4 &yp,
                                        const Pair4 &zm, const Pair4 &zp, uint32_t below) {
                        // outside the box at both ends of a row: not used there
                        const float l = s[r][x - 1], rt = s[r][x + 4];
                        o.cl = cd[r][15 + x];
                        if (!listed(o, below)) {
                            const uint32_t m = media(o.c);
                            return fma4(entry(tw, m), neighbours(c, l, rt, ym, yp, zm, zp), mul4(entry(td, m), c));
                        }
                        Pair4 sum, dg;
                        listed_sums(cp, L, q, o, below, c, l, rt, ym, yp, zm, zp, sum, dg);
                        return fma4(OMEGA, sum, mul4(scale(1.f - OMEGA, dg), c));
                    };
                    o.c = nbA;
                    o.cy = word(cd, ra - 1);
                    rA = residual(p, ra, cA, p4(f4(&s[ra - 1][x])), cB, mA, nA, bA);
                    if (rowB) {
                        o.c = nbB;
                        o.cy = nbA;
                        rB = residual(p + L.sx, ra + 1, cB, cA, p4(f4(&s[ra + 2][x])), mB, nB, bB);
                    }
                    if (edge) {
                        clip(rA);
                        clip(rB);
                    }
                }
                const Pair4 h = scale(0.5f, rA);
                next = h + rB;
                if (work) {
                    *reinterpret_cast<float4 *>(&half[ODD][pr][x]) = f4(h);
                    last[ODD][pr][u] = next.b.y;
                }
                mA = cA;
                mB = cB;
                cA = nA;
                cB = nB;
                bA = nbA;
                bB = nbB;
            }
            if (k > ka && pr < C0Y) {  // restrict plane k - 1
                const float *h = half[!ODD][pr + 1] + x;
                const Pair4 y = share + p4(f4(h));
                const float left = u > 0 ? last[!ODD][pr][u - 1] + h[-1] : 0.f;
                const float t0 = y.a.x + 0.5f * (left + y.a.y), t1 = y.b.x + 0.5f * (y.a.y + y.b.y);
                if (ODD) {
                    acc0 += t0;
                    acc1 += t1;
                } else {
                    if (done && in0) C.s[pc] = __fdividef(acc0 + 0.5f * t0, dc0);
                    if (done && in1) C.s[pc + 1] = __fdividef(acc1 + 0.5f * t1, dc1);
                    acc0 = 0.5f * t0;
                    acc1 = 0.5f * t1;
                }
            }
            share = next;
        };
        for (int k = ka; k <= kb; k += 2) {
            step(k, std::true_type{}, true);
            step(k + 1, std::false_type{}, k + 1 <= kb);
        }
        ring.report(e.st);
    }
}

// Correction, post-smoothing and rho of level 0.  Warps 0 to 3 own the tile's
// eight row pairs (an odd row and the even one above), warp 4 the row on
// either side, warp 5 the column on either side; all put v = omega s + P e in
// shared memory, three planes deep.  Planes are taken in pairs, as a coarse
// plane serves two of them; its tile comes in by asynchronous copies.
template <bool SINGLE>
__global__ void __launch_bounds__(mg::U0NT, 3)
k_mg_up0(const mg::Entry *__restrict__ tab, mg::Head *__restrict__ head, int total,
         const __grid_constant__ mg::Entry e0) {
    using namespace mg;
    using R = Ring<U0R, U0W, FY + 1>;
    // a row: column i0 - 1 at [3], i0 .. i0 + 63 from [4], i0 + 64 at [68]
    constexpr int NT = U0NT, VW = U0W, CZX = FX / 2 + 8, CZY = FY / 2 + 2, CZU = CZX / 4;
    __shared__ __align__(16) float vp[3][FY + 2][VW];
    __shared__ __align__(128) R::Mem planes;
    __shared__ __align__(16) float cz[3][CZY][CZX];  // coarse planes: columns i0 / 2 - 4 .., rows (j0 - 1) / 2 ..
    __shared__ float4 tq[16], td[16];                // omega w / d and d
    __shared__ float sred[2][4];
    __shared__ uint64_t bars[NS];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int u = lane & 15, hi = lane >> 4;
    const bool own = w < 4, hrow = w == 4;
    // row (0 .. FY + 1; own threads: their first) and column of vp and ss
    const int r = own ? 1 + 4 * w + 2 * hi : (hrow ? (hi ? FY + 1 : 0) : 1 + u);
    const int x = own || hrow ? 4 + 4 * u : (hi ? 4 + FX : 3);
    R ring(planes, bars);
    // a limit of no polls gives up before anything is issued: a wait looks at
    // its slot once before it counts
    const bool no_polls = tma::g_slot_wait_limit == 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int nsys = SINGLE ? 1 : head->nsys;
    if (!SINGLE) total = head->utotal[0];
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        const Entry &e = SINGLE ? e0 : tab[find_sys(tab, nsys, it, &Entry::ubase, 0)];
        // one answer for the block; and the previous item's last reads, the barriers' initialisation
        if (__syncthreads_or(*(volatile int *)&e.st->done | (int)no_polls)) {
            if (no_polls) ring.fail(e.st);
            continue;
        }
        const Lev L = e.lev[0], C = e.lev[1];
        const CoefC32 cp = e.cp;
        float *const partials = e.partials;
        const bool padded = e.nbot > 1;
        const int li = SINGLE ? it : it - e.ubase[0];
        const int xt = (L.nx - 1 + FX - 1) / FX, yt = (L.ny - 2 + FY - 1) / FY;
        const int col = li % (xt * yt), ch = li / (xt * yt);
        const int i0 = (col % xt) * FX, j0 = 1 + (col / xt) * FY;
        const int k0 = 1 + ch * e.uk[0], k1 = min(k0 + e.uk[0], L.nz - 1);  // k0 odd
        const int j = j0 - 1 + r, ib = i0 - 4 + x;
        const bool cols = ib >= 0 && ib <= L.nx - 2;
        const bool rowA = cols && j >= 1 && j <= L.ny - 2, rowB = own && rowA && j + 1 <= L.ny - 2;
        const int pj = j * L.sx + ib;
        const bool edge = ib < 1 || ib + 3 > L.nx - 2;
        auto clip = [&](Pair4 &v) {  // columns that are no unknowns
            if (ib < 1) v.a.x = 0.f;
            if (ib + 1 > L.nx - 2) v.a.y = 0.f;
            if (ib + 2 > L.nx - 2) v.b.x = 0.f;
            if (ib + 3 > L.nx - 2) v.b.y = 0.f;
        };
        // a coarse plane's tile into slot K % 3: a unit a thread
        const int cu = tid % CZU, cv = tid / CZU;
        const int Ic = i0 / 2 - 4 + 4 * cu, Jc = (j0 - 1) / 2 + cv;
        const bool cin = cv < CZY && Ic >= 0 && Ic < C.sx && Jc < C.ny;
        auto fetch_coarse = [&](int K) {
            if (cv < CZY) {
                const bool in = cin && K < C.nz;
                const float *src = C.z + (in ? K * C.sxy + Jc * C.sx + Ic : 0);
                float *dst = &cz[K % 3][cv][4 * cu];
                if (padded) {
                    cp_async16(dst, src, in);
                } else {  // the bottom kernel's rows are not padded
                    for (int q = 0; q < 4; ++q) {
                        const bool t = in && Ic + q < C.nx;
                        cp_async4(dst + q, t ? src + q : C.z, t);
                    }
                }
            }
        };
        // coarse correction of plane K at the thread's nodes, interpolated in x
        // and y: of its first row (or node), and of the row above
        struct E2 {
            Pair4 a, b;
        };
        const int ca = (j >> 1) - (j0 - 1) / 2, cb = ((j + 1) >> 1) - (j0 - 1) / 2, ci = (ib >> 1) - i0 / 2 + 4;
        auto coarse = [&](int K) {
            E2 t = {};
            const float *a = &cz[K % 3][ca][ci], *b = &cz[K % 3][cb][ci];
            if (own || hrow) {
                const float2 b01 = *reinterpret_cast<const float2 *>(b), a01 = *reinterpret_cast<const float2 *>(a);
                const float b2 = b[2], a2 = 0.5f * (a[2] + b2);
                const float a0 = 0.5f * (a01.x + b01.x), a1 = 0.5f * (a01.y + b01.y);
                t.a = {make_float2(a0, 0.5f * (a0 + a1)), make_float2(a1, 0.5f * (a1 + a2))};
                t.b = {make_float2(b01.x, 0.5f * (b01.x + b01.y)), make_float2(b01.y, 0.5f * (b01.y + b2))};
            } else {
                const int o = ib & 1;  // an odd column lies between two coarse ones
                t.a.a.x = 0.25f * ((a[0] + a[o]) + (b[0] + b[o]));
            }
            return t;
        };
        // v = omega s + P e of plane k, into vp[slot]
        Pair4 vA, vB;  // the last one made (own rows)
        auto make_v = [&](int k, int slot, const E2 &g) {  // of the last plane waited for
            vA = vB = Pair4{};
            const bool kin = k >= 1 && k <= L.nz - 2;
            const float (*s)[VW] = ring.s(0);
            if (own || hrow) {
                if (rowA && kin) {
                    vA = fma4(OMEGA, p4(f4(&s[r][x])), g.a);
                    if (rowB) vB = fma4(OMEGA, p4(f4(&s[r + 1][x])), g.b);
                    if (edge) {
                        clip(vA);
                        clip(vB);
                    }
                }
                *reinterpret_cast<float4 *>(&vp[slot][r][x]) = f4(vA);
                if (own) *reinterpret_cast<float4 *>(&vp[slot][r + 1][x]) = f4(vB);
            } else {
                vp[slot][r][x] = rowA && kin ? OMEGA * s[r][x] + g.a.a.x : 0.f;
            }
        };
        auto mean = [](const E2 &p, const E2 &q) { return E2{scale(0.5f, p.a + q.a), scale(0.5f, p.b + q.b)}; };
        const int first = min(4, k1 - k0 + 2);  // planes to begin with
        for (int q = 0; q < first; ++q) ring.issue(e.su, e.cu, i0, j0 - 1, k0 - 1 + q, q);
        for (int K = (k0 - 1) >> 1; K <= (k0 + 3) >> 1; ++K) fetch_coarse(K);
        if (tid < 16) fill_media(tq, tid, __fdividef(OMEGA * cp.w_in, e.dg_in), __fdividef(OMEGA * cp.w_out, e.dg_out));
        else if (tid < 32) fill_media(td, tid - 16, e.dg_in, e.dg_out);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        E2 ec = coarse((k0 - 1) >> 1), en = coarse((k0 + 1) >> 1);
        int slot = (k0 - 1) % 3;  // of plane k - 1
        ring.wait(first - 1);
        make_v(k0 - 1, slot, ec);
        Pair4 mA = vA, mB = vB;
        ring.wait(first - 2);
        make_v(k0, slot == 2 ? 0 : slot + 1, mean(ec, en));
        Pair4 cA = vA, cB = vB;
        ec = en;  // coarse plane (k0 + 1) / 2
        auto word = [&](const uint8_t (*c)[C0W], int q) { return *reinterpret_cast<const uint32_t *>(&c[q][12 + x]); };
        uint32_t bA = 0, bB = 0;  // codes of plane k - 1
        if (own) {
            bA = word(ring.c(1), r);
            bB = word(ring.c(1), r + 1);
        }
        // rho: every RG planes of a tile have a partial of their own, so that
        // the sum does not depend on the planes per work item (uk[0] is a
        // multiple of RG).  The one that ends with plane k is written here,
        // a barrier after the warps' sums.
        auto flush = [&](int k) {
            const float *q = sred[((k - 1) / RG) & 1];
            partials[((k - 1) / RG) * xt * yt + col] = ((q[0] + q[1]) + q[2]) + q[3];
        };
        Pair4 rho = {};
        // one plane: v(k + 1) with the correction g, then z(k)
        auto step = [&](int k, const E2 &g) {
            const int sv = slot == 2 ? 0 : slot + 1, sn = sv == 2 ? 0 : sv + 1;
            ring.wait(k + 2 <= k1);  // plane k + 1
            make_v(k + 1, sn, g);
            const Pair4 nA = vA, nB = vB;
            __syncthreads();
            if (k + 3 <= k1) ring.issue(e.su, e.cu, i0, j0 - 1, k + 3, 1);  // over plane k - 1
            if (tid == 0 && k > k0 && (k - 1) % RG == 0) flush(k - 1);
            if (own) {
                uint32_t nbA = 0, nbB = 0;
                if (rowA) {
                    const float (*v)[VW] = vp[sv];
                    const float (*ss)[VW] = ring.s(1);
                    const uint8_t (*cd)[C0W] = ring.c(1);
                    nbA = word(cd, r);
                    nbB = word(cd, r + 1);
                    Codes o;
                    auto relax = [&](int q, const Pair4 &s, const Pair4 &c, int rr, const Pair4 &ym, const Pair4 &yp,
                                     const Pair4 &zm, const Pair4 &zp, uint32_t below) {
                        const float l = v[rr][x - 1], rt = v[rr][x + 4];
                        o.cl = cd[rr][11 + x];
                        Pair4 z = fma4(1.f - OMEGA, c, scale(OMEGA, s)), d;
                        if (!listed(o, below)) {
                            const uint32_t m = media(o.c);
                            d = entry(td, m);
                            z = fma4(entry(tq, m), neighbours(c, l, rt, ym, yp, zm, zp), z);
                        } else {
                            Pair4 sum;
                            listed_sums(cp, L, q, o, below, c, l, rt, ym, yp, zm, zp, sum, d);
                            z = fma4(OMEGA,
                                     Pair4{make_float2(__fdividef(sum.a.x, d.a.x), __fdividef(sum.a.y, d.a.y)),
                                           make_float2(__fdividef(sum.b.x, d.b.x), __fdividef(sum.b.y, d.b.y))},
                                     z);
                        }
                        if (edge) clip(z);
                        rho = fma4(mul4(d, s), z, rho);
                        *reinterpret_cast<float4 *>(L.z + q) = f4(z);
                    };
                    const int p = k * L.sxy + pj;
                    o.c = nbA;
                    o.cy = word(cd, r - 1);
                    relax(p, p4(f4(&ss[r][x])), cA, r, p4(f4(&v[r - 1][x])), cB, mA, nA, bA);
                    if (rowB) {
                        o.c = nbB;
                        o.cy = nbA;
                        relax(p + L.sx, p4(f4(&ss[r + 1][x])), cB, r + 1, cA, p4(f4(&v[r + 2][x])), mB, nB, bB);
                    }
                }
                if (k % RG == 0 || k == k1 - 1) {
                    const float t = tma::warp_sum_f((rho.a.x + rho.a.y) + (rho.b.x + rho.b.y));
                    if (lane == 0) sred[((k - 1) / RG) & 1][w] = t;
                    rho = Pair4{};
                }
                mA = cA;
                mB = cB;
                cA = nA;
                cB = nB;
                bA = nbA;
                bB = nbB;
            }
            slot = sv;
        };
        for (int k = k0; k < k1; k += 2) {
            asm volatile("cp.async.wait_all;" ::: "memory");  // coarse plane (k + 3) / 2: behind the next barrier
            step(k, ec);                                      // v(k + 1): an even plane, coarse plane (k + 1) / 2
            if (k + 1 >= k1) break;
            fetch_coarse((k + 5) >> 1);
            en = coarse((k + 3) >> 1);
            step(k + 1, mean(ec, en));
            ec = en;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (tid == 0) flush(k1 - 1);
        ring.report(e.st);
    }
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

// What the bottom kernel keeps in shared memory besides its vectors, made with
// the hierarchy: for every node of its levels, one after the other and
// unpadded, the weights and the diagonal (arrays of T values); for every
// interior node, its place in its level, its parent (the coarse node below it
// and the three parities) and, on coarse levels, its fine node.
template <class E>
__global__ void k_mg_pack(const __grid_constant__ E e, int T) {
    using namespace mg;
    using F = typename E::T;
    F *W = reinterpret_cast<F *>(e.blob);
    uint16_t *list = reinterpret_cast<uint16_t *>(W + 4 * T), *up = list + T, *dn = up + T;
    int off = 0;
    for (int l = e.nbot; l < e.nlev; ++l) {
        const auto &L = e.lev[l];
        const int n = L.nx * L.ny * L.nz, mx = L.nx - 2, my = L.ny - 2;
        const int cx = L.nx / 2 + 1, cxy = cx * (L.ny / 2 + 1);
        const int fx = l > e.nbot ? e.lev[l - 1].nx : 0, fxy = l > e.nbot ? fx * e.lev[l - 1].ny : 0;
        for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
            W[off + p] = L.wx[p];
            W[T + off + p] = L.wy[p];
            W[2 * T + off + p] = L.wz[p];
            W[3 * T + off + p] = L.dg[p];
            const int i = p % L.nx, j = (p / L.nx) % L.ny, k = p / (L.nx * L.ny);
            if (!interior(L, i, j, k)) continue;
            const int t = off + ((k - 1) * my + j - 1) * mx + i - 1;
            list[t] = (uint16_t)p;
            up[t] = (uint16_t)((((k >> 1) * cxy + (j >> 1) * cx + (i >> 1)) << 3) | ((k & 1) << 2) | ((j & 1) << 1) |
                               (i & 1));
            dn[t] = (uint16_t)(2 * k * fxy + 2 * j * fx + 2 * i);
        }
        off += n;
    }
}

// The levels nbot .. nlev - 1 of one system per block, in shared memory.  The
// same cycle as above; SWEEPS damped Jacobi steps on the last level.  One SM
// works here, and what it does serially counts: the coefficients and node lists come in
// one asynchronous copy, before the previous kernel has ended (one-system
// launches).
template <class E, bool SINGLE>
__global__ void __launch_bounds__(mg::BOT_T, 1)
k_mg_bottom(const E *__restrict__ tab, const mg::Head *__restrict__ head,
            const __grid_constant__ E e0) {
    using namespace mg;
    using F = typename E::T;
    constexpr F OM = OMEGA;
    extern __shared__ __align__(16) char bsm[];
    const int tid = threadIdx.x;
    if (!SINGLE) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if ((int)blockIdx.x >= head->nsys) return;
    }
    const E &e = SINGLE ? e0 : tab[blockIdx.x];
    const int lb = e.nbot, le = e.nlev, T = e.bot;
    if (le == 0) return;
    if (!SINGLE && *(volatile int *)&e.st->done) return;
    const F *Wx = reinterpret_cast<const F *>(bsm), *Wy = Wx + T, *Wz = Wy + T, *D = Wz + T;
    const uint16_t *list = reinterpret_cast<const uint16_t *>(D + T), *up = list + T, *dn = up + T;
    F *S = reinterpret_cast<F *>(bsm + BLOB_BYTES<F> * T), *Z = S + T, *R = Z + T;
    // T is a multiple of 8, so the blob is whole 16-byte pieces.  Not of a solve
    // that has ended: the engine hands its system back while a replay that
    // holds it may still be in flight, and its memory may be gone by then.
    const bool ended = SINGLE && *(volatile int *)&e.st->done;
    for (int q = ended ? INT_MAX : tid; q < BLOB_BYTES<F> * T / 16; q += BOT_T)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tma::smem_u32(bsm + 16 * q)),
                     "l"(reinterpret_cast<const char *>(e.blob) + 16 * q)
                     : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int q = tid; q < 3 * T; q += BOT_T) S[q] = 0;
    if (SINGLE) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    const bool skip = ended || (SINGLE && *(volatile int *)&e.st->done);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (skip) return;
    __syncthreads();
    {
        const auto &L = e.lev[lb];
        const int n = L.nx * L.ny * L.nz;
#pragma unroll 8
        for (int p = tid; p < n; p += BOT_T) S[p] = L.s[p];
    }
    __syncthreads();
    // sum over the faces of node p of the level whose nodes start at o
    auto faces = [&](int o, int sx, int sxy, const F *x, int p) {
        const F *a = Wx + o, *b = Wy + o, *c = Wz + o;
        return ((a[p - 1] * x[p - 1] + a[p] * x[p + 1]) + (b[p - sx] * x[p - sx] + b[p] * x[p + sx])) +
               (c[p - sxy] * x[p - sxy] + c[p] * x[p + sxy]);
    };
    int o = 0;
    for (int l = lb; l < le - 1; ++l) {
        const auto &L = e.lev[l], &C = e.lev[l + 1];
        const int sx = L.nx, sxy = L.nx * L.ny, n = (L.nx - 2) * (L.ny - 2) * (L.nz - 2);
        const int oc = o + sxy * L.nz, nc = (C.nx - 2) * (C.ny - 2) * (C.nz - 2);
        for (int t = tid; t < n; t += BOT_T) {
            const int p = list[o + t];
            R[o + p] = ((F)1 - OM) * D[o + p] * S[o + p] + OM * faces(o, sx, sxy, S + o, p);
        }
        __syncthreads();
        for (int t = tid; t < nc; t += BOT_T) {
            const int pc = list[oc + t];
            const F *f = R + o + dn[oc + t];
            F acc = 0.f;
#pragma unroll
            for (int c = -1; c <= 1; ++c)
#pragma unroll
                for (int b = -1; b <= 1; ++b) {
                    const F *x = f + c * sxy + b * sx;
                    acc += (b ? (F)0.5 : (F)1) * (c ? (F)0.5 : (F)1) * (x[0] + (F)0.5 * (x[-1] + x[1]));
                }
            S[oc + pc] = quotient(acc, D[oc + pc]);
        }
        __syncthreads();
        o = oc;
    }
    {
        const auto &L = e.lev[le - 1];
        const int sx = L.nx, sxy = L.nx * L.ny, n = (L.nx - 2) * (L.ny - 2) * (L.nz - 2);
        if (n == 1) {  // one unknown: its solution
            if (tid == 0) Z[o + list[o]] = S[o + list[o]];
        } else {
            F *a = Z + o, *b = R + o;
            for (int t = tid; t < n; t += BOT_T) a[list[o + t]] = OM * S[o + list[o + t]];
            __syncthreads();
            for (int q = 1; q < SWEEPS; ++q) {
                for (int t = tid; t < n; t += BOT_T) {
                    const int p = list[o + t];
                    b[p] = ((F)1 - OM) * a[p] +
                           OM * (S[o + p] + quotient(faces(o, sx, sxy, a, p), D[o + p]));
                }
                __syncthreads();
                F *t = a;
                a = b;
                b = t;
            }
            if (a != Z + o)
                for (int t = tid; t < n; t += BOT_T) Z[o + list[o + t]] = a[list[o + t]];
        }
        __syncthreads();
    }
    for (int l = le - 2; l >= lb; --l) {
        const auto &L = e.lev[l], &C = e.lev[l + 1];
        const int sx = L.nx, sxy = L.nx * L.ny, n = (L.nx - 2) * (L.ny - 2) * (L.nz - 2);
        const int cx = C.nx, cxy = C.nx * C.ny, oc = o;
        o -= sxy * L.nz;
        for (int t = tid; t < n; t += BOT_T) {
            const int p = list[o + t], c = up[o + t];
            const F *x = Z + oc + (c >> 3);
            const int di = c & 1, dj = (c & 2) ? cx : 0, dk = (c & 4) ? cxy : 0;
            const F acc = ((x[0] + x[di]) + (x[dj] + x[dj + di])) + ((x[dk] + x[dk + di]) + (x[dk + dj] + x[dk + dj + di]));
            R[o + p] = OM * S[o + p] + (F)0.125 * acc;
        }
        __syncthreads();
        for (int t = tid; t < n; t += BOT_T) {
            const int p = list[o + t];
            const F z = ((F)1 - OM) * R[o + p] +
                            OM * (S[o + p] + quotient(faces(o, sx, sxy, R + o, p), D[o + p]));
            Z[o + p] = z;
        }
        __syncthreads();
    }
    const auto &L = e.lev[lb];
    for (int p = tid; p < L.nx * L.ny * L.nz; p += BOT_T) L.z[p] = Z[p];
}

// Edge weights and ionic term (kept in z while the hierarchy is built) of a
// coarse level: from the FP64 weights and the code bytes of level 0, or
// from a coarse level.
template <bool FINE, typename T>
__global__ void k_mg_coarsen(mg::LevT<T> F, mg::LevT<T> C, const double *__restrict__ Wx, const double *__restrict__ Wy,
                             const double *__restrict__ Wz, const uint8_t *__restrict__ code, T kap0) {
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t >= C.nx * C.ny * C.nz) return;
    const int I = t % C.nx, J = (t / C.nx) % C.ny, K = t / (C.nx * C.ny);
    const int n[3] = {F.nx, F.ny, F.nz}, c[3] = {I, J, K};
    auto weight = [&](int d, const int (&x)[3]) -> T {
        if (FINE) {
            const double *W = d == 0 ? Wx : (d == 1 ? Wy : Wz);
            return (T)W[((long long)x[2] * F.ny + x[1]) * F.nx + x[0]];
        }
        return (d == 0 ? F.wx : (d == 1 ? F.wy : F.wz))[x[2] * F.sxy + x[1] * F.sx + x[0]];
    };
    T W[3];
    for (int d = 0; d < 3; ++d) {
        const int u = (d + 1) % 3, v = (d + 2) % 3;
        T sum = (T)0;
        for (int b = -1; b <= 1; ++b)
            for (int a = -1; a <= 1; ++a) {
                int x[3];
                x[u] = min(max(2 * c[u] + a, 0), n[u] - 1);
                x[v] = min(max(2 * c[v] + b, 0), n[v] - 1);
                x[d] = min(2 * c[d], n[d] - 2);
                const T p = weight(d, x);
                T w;
                if (2 * c[d] + 1 <= n[d] - 2) {
                    x[d] += 1;
                    const T q = weight(d, x);
                    w = (T)0.5 * (p * (q / (p + q)) + (T)0.25 * (p + q));  // p q may leave the range of the type
                } else {
                    w = p;  // one fine edge to the boundary
                }
                sum += (a ? (T)0.5 : (T)1) * (b ? (T)0.5 : (T)1) * w;
            }
        W[d] = c[d] < (d == 0 ? C.nx : (d == 1 ? C.ny : C.nz)) - 1 ? sum : (T)0;
    }
    T kap = (T)0;
    for (int e = 0; e < 27; ++e) {
        const int a = e % 3 - 1, b = (e / 3) % 3 - 1, g = e / 9 - 1;
        const int x = min(max(2 * I + a, 0), F.nx - 1), y = min(max(2 * J + b, 0), F.ny - 1),
                  z = min(max(2 * K + g, 0), F.nz - 1);
        const int p = z * F.sxy + y * F.sx + x;
        const T k = FINE ? ((code[p] & 1) ? (T)0 : kap0) : F.z[p];
        kap += (a ? (T)0.5 : (T)1) * (b ? (T)0.5 : (T)1) * (g ? (T)0.5 : (T)1) * k;
    }
    const int p = K * C.sxy + J * C.sx + I;
    C.wx[p] = W[0];
    C.wy[p] = W[1];
    C.wz[p] = W[2];
    if (C.dg) C.dg[p] = (T)1;
    C.z[p] = kap;
}

template <typename T>
__global__ void k_mg_diag(mg::LevT<T> C) {
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t >= C.nx * C.ny * C.nz) return;
    const int I = t % C.nx, J = (t / C.nx) % C.ny, K = t / (C.nx * C.ny);
    if (!mg::interior(C, I, J, K)) return;
    const int p = K * C.sxy + J * C.sx + I;
    const T d = C.wx[p] + C.wx[p - 1] + C.wy[p] + C.wy[p - C.sx] + C.wz[p] + C.wz[p - C.sxy] + C.z[p];
    C.dg[p] = d;
    if (C.di) C.di[p] = (T)1 / d;
}

// The FP64 cycle (plain FP64 solver): the same steps with stored weights and
// 1 / diagonal on every level, a node a thread.  GB300's FP64 pipe binds these
// kernels before memory does (about 50 FP64 operations per unknown and cycle),
// so residual, restriction, interpolation and smoothing are kernels of their
// own and no value is formed twice.  97^3 to 1e-12: 500 Jacobi iterations and
// 29.9 ms -> 29 iterations and 5.9 ms (7.3 ms with a node a thread in the top smoother, whose block sums
// then cost as much as its stencil, with divisions in the bottom kernel and
// without programmatic launches).
namespace mg {
struct Entry64 {
    using T = double;
    LevT<double> lev[LMAX];
    int nlev, nbot;
    CgState *st;
    void *blob;
    int bot;
};
__device__ __forceinline__ double face_sum64(const LevT<double> &L, const double *x, int p) {
    return ((L.wx[p - 1] * x[p - 1] + L.wx[p] * x[p + 1]) + (L.wy[p - L.sx] * x[p - L.sx] + L.wy[p] * x[p + L.sx])) +
           (L.wz[p - L.sxy] * x[p - L.sxy] + L.wz[p] * x[p + L.sxy]);
}
// interior node t
__device__ __forceinline__ bool node64(const LevT<double> &L, int t, int &i, int &j, int &k) {
    const int mx = L.nx - 2, my = L.ny - 2;
    if (t >= mx * my * (L.nz - 2)) return false;
    const int r = t / mx;
    i = 1 + t - r * mx;
    k = 1 + r / my;
    j = 1 + r - (k - 1) * my;
    return true;
}
}  // namespace mg

__global__ void __launch_bounds__(256) k_mg64_residual(mg::LevT<double> L, const CgState *st) {
    using namespace mg;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*(volatile const int *)&st->done) return;
    int i, j, k;
    if (!node64(L, blockIdx.x * 256 + threadIdx.x, i, j, k)) return;
    const int p = k * L.sxy + j * L.sx + i;
    L.r[p] = (1.0 - (double)OMEGA) * L.dg[p] * L.s[p] + (double)OMEGA * face_sum64(L, L.s, p);
}

__global__ void __launch_bounds__(256) k_mg64_restrict(mg::LevT<double> L, mg::LevT<double> C, const CgState *st) {
    using namespace mg;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*(volatile const int *)&st->done) return;
    int I, J, K;
    if (!node64(C, blockIdx.x * 256 + threadIdx.x, I, J, K)) return;
    const double *f = L.r + (2 * K * L.sxy + 2 * J * L.sx + 2 * I);
    double acc = 0.0;
#pragma unroll
    for (int c = -1; c <= 1; ++c)
#pragma unroll
        for (int b = -1; b <= 1; ++b) {
            const double *x = f + c * L.sxy + b * L.sx;
            acc += (b ? 0.5 : 1.0) * (c ? 0.5 : 1.0) * (x[0] + 0.5 * (x[-1] + x[1]));
        }
    const int p = K * C.sxy + J * C.sx + I;
    C.s[p] = acc * C.di[p];
}

__global__ void __launch_bounds__(256) k_mg64_correct(mg::LevT<double> L, mg::LevT<double> C, const CgState *st) {
    using namespace mg;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*(volatile const int *)&st->done) return;
    int i, j, k;
    if (!node64(L, blockIdx.x * 256 + threadIdx.x, i, j, k)) return;
    // an even coordinate lies on a coarse line: no sum along it.  The values of
    // the corners are added up and scaled once.
    const double *x = C.z + ((k >> 1) * C.sxy + (j >> 1) * C.sx + (i >> 1));
    const bool odd = i & 1;
    auto line = [&](const double *q) { return odd ? q[0] + q[1] : q[0]; };
    auto plane = [&](const double *q) { return (j & 1) ? line(q) + line(q + C.sx) : line(q); };
    const double e = (k & 1) ? plane(x) + plane(x + C.sxy) : plane(x);
    const double f = __hiloint2double(0x3FF00000 - (((i & 1) + (j & 1) + (k & 1)) << 20), 0);  // 2^-(odd coordinates)
    const int p = k * L.sxy + j * L.sx + i;
    L.r[p] = fma(f, e, (double)OMEGA * L.s[p]);
}

// the post-smoothing step (v in r); level 0: rho = r.z and beta
template <bool TOP>
__global__ void __launch_bounds__(256) k_mg64_smooth(mg::LevT<double> L, CgState *st, double *partials) {
    using namespace mg;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*(volatile const int *)&st->done) return;
    __shared__ double sred[8];
    int i, j, k;
    double rho = 0.0;
    // level 0: several nodes a thread, as the block's sum takes six FP64
    // operations a warp and value
    for (int t = blockIdx.x * 256 + threadIdx.x; node64(L, t, i, j, k); t += gridDim.x * 256) {
        const int p = k * L.sxy + j * L.sx + i;
        const double s = L.s[p];
        const double z = (1.0 - (double)OMEGA) * L.r[p] + (double)OMEGA * (s + face_sum64(L, L.r, p) * L.di[p]);
        L.z[p] = z;
        if (!TOP) return;
        rho = fma(L.dg[p] * s, z, rho);
    }
    if (!TOP) return;  // a thread without a node
    double t0, t1;
    if (last_block_total<256, false>(st, partials, gridDim.x, rho, 0.0, sred, t0, t1) && threadIdx.x == 0) {
        st->counter = 0;
        if (!(t0 > 0.0) || !isfinite(t0)) {
            st->done = 1;
            st->status = 1;
        } else {
            st->beta = st->rho > 0.0 ? t0 / st->rho : 0.0;
            st->rho = t0;
        }
    }
}

// ------------------------------------------------------------------- host --
struct MgState {
    mg::Entry e{};
    mg::Head *head = nullptr;    // device, of one-system launches
    float *v = nullptr;          // preconditioned residual (padded, level 0)
    void *mem = nullptr;         // coarse levels
    bool lattice = false;        // level 0 has stored coefficients too
    float *partials = nullptr;
};

// Planes per work item.  A block marches over them after reading two more,
// at about a microsecond a plane: the count with the fewest rounds of blocks
// times planes, by the blocks that share an SM (level 0 of a solver's grid four
// down and three up, stored levels three and two.  Counted as four and three
// there too, the stored 129^3 level took a second round for some blocks: 257^3
// 13.31 -> 12.93 ms, 150 x 97 x 118 3.82 -> 3.75 ms, others the same).
// shared: many systems fill the launch, and the longest items waste least.
// Only the work is divided differently, the results are the same bits.
void mg_planes(mg::Entry &e, bool shared) {
    using namespace mg;
    auto best = [&](long long cols, int n, int slots, int step, int most) {
        int kc = most;
        double cost = 1e30;
        const int longest = shared ? 0 : most;
        for (int c = step; c <= longest; c += step) {
            const double t = (double)cdiv(cols * cdiv(n, c), (long long)slots * num_sms()) * (c + 2.5);
            if (t < cost) {
                cost = t;
                kc = c;
            }
        }
        return kc;
    };
    for (int l = 0; l < e.nbot; ++l) {
        const Lev &F = e.lev[l], &C = e.lev[l + 1];
        // a coarse plane is two fine ones
        e.dk[l] = best((long long)cdiv(C.nx - 2, CX) * cdiv(C.ny - 2, l == 0 && e.code ? C0Y : CY), 2 * (C.nz - 2),
                       l == 0 && e.code ? 4 : 3, 2, 16) / 2;
        e.uk[l] = best((long long)cdiv(F.nx - 1, FX) * cdiv(F.ny - 2, FY), F.nz - 2,
                       l == 0 && e.code ? 3 : 2, l == 0 ? RG : 1, 16);
    }
}

// The levels of a grid; false when the hierarchy does not reach the bottom
// kernel's size (grids thinner than 9 nodes, or very long and thin ones):
// those keep the Jacobi preconditioner.
template <class E>
bool mg_levels(const PadGeo &g, E &e, bool lattice = false) {
    using namespace mg;
    if (std::min(g.nx, std::min(g.ny, g.nz)) < 9) return false;
    int n[3] = {g.nx, g.ny, g.nz}, nl = 0;
    for (;; ++nl) {
        if (nl == LMAX) return false;
        LevT<typename E::T> &L = e.lev[nl];
        L = LevT<typename E::T>{};
        L.nx = n[0];
        L.ny = n[1];
        L.nz = n[2];
        L.sx = nl == 0 && !lattice ? g.sx : ((n[0] + 3) & ~3);
        L.sxy = L.sx * n[1];
        if (std::min(n[0], std::min(n[1], n[2])) < 5) break;
        for (int d = 0; d < 3; ++d) n[d] = n[d] / 2 + 1;
    }
    e.nlev = nl + 1;
    long long nodes = 0;
    int b = e.nlev;
    while (b > (lattice ? 0 : 1)) {  // level 0 of a solver's grid is not the bottom kernel's
        const auto &L = e.lev[b - 1];
        const long long n = (long long)L.nx * L.ny * L.nz;
        if (nodes + n > BOT_NODES<typename E::T>) break;
        nodes += n;
        --b;
    }
    if (b == e.nlev) return false;
    e.nbot = b;
    e.bot = (int)((nodes + 7) & ~7ll);
    for (int l = b; l < e.nlev; ++l) {
        e.lev[l].sx = e.lev[l].nx;
        e.lev[l].sxy = e.lev[l].nx * e.lev[l].ny;
    }
    if constexpr (std::is_same<E, Entry>::value) {
        const Lev &F = e.lev[0];
        if (!lattice) e.nu0 = cdiv(F.nx - 1, FX) * cdiv(F.ny - 2, FY) * cdiv(F.nz - 2, RG);
        mg_planes(e, false);
    }
    return true;
}

// elements of one array of a level (whole 16-byte pieces)
template <typename T>
size_t mg_lev_size(const mg::LevT<T> &L) { return ((size_t)L.sxy * L.nz + 3) & ~(size_t)3; }

void mg_release(MgState *m, cudaStream_t s) {
    if (!m) return;
    dfree(m->head, s);
    dfree(m->v, s);
    dfree(m->mem, s);
    dfree(m->partials, s);
    delete m;
}

void free_mg_state(pb_system *sys) {
    mg_release((MgState *)sys->mg, sys->stream);
    sys->mg = nullptr;
}

template <class E>
size_t mg_bottom_bytes(const E &e) {
    return (size_t)mg::BOT_BYTES<typename E::T> * e.bot;
}

// attributes of the bottom kernels on the current device (set again with every
// hierarchy and engine: nothing is remembered across threads and devices)
pb_status mg_prepare() {
    const int most = mg::BOT_BYTES<float> * mg::BOT_NODES<float>, most64 = mg::BOT_BYTES<double> * mg::BOT_NODES<double>;
    PB_CUDA_TRY(cudaFuncSetAttribute(k_mg_bottom<mg::Entry, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    PB_CUDA_TRY(cudaFuncSetAttribute(k_mg_bottom<mg::Entry, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    PB_CUDA_TRY(
        cudaFuncSetAttribute(k_mg_bottom<mg::Entry64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most64));
    return PB_OK;
}

// lays the arrays of levels first .. nlev - 1 and the bottom kernel's data out
// in `base`; returns the bytes (base may be null)
template <class E>
size_t mg_layout(E &e, int first, char *base) {
    using T = typename E::T;
    constexpr int arrays = sizeof(T) == 4 ? 6 : 8;
    size_t at = 0;
    for (int l = first; l < e.nlev; ++l) {
        mg::LevT<T> &L = e.lev[l];
        const size_t n = mg_lev_size(L);
        if (base) {
            L.wx = (T *)(base + at);  // n is a multiple of 4: every array is 16-byte aligned
            L.wy = L.wx + n;
            L.wz = L.wy + n;
            L.dg = L.wz + n;
            L.s = L.dg + n;
            L.z = L.s + n;
            if (arrays == 8) {
                L.di = L.z + n;
                L.r = L.di + n;
            }
        }
        at += n * arrays * sizeof(T);
    }
    if (base) e.blob = base + at;
    return at + mg::BLOB_BYTES<T> * (size_t)e.bot;
}

// coefficients of levels first .. nlev - 1 from the level above (level 1 of a
// solver's grid from its FP64 operator; first == 0: level 0 is there already,
// its ionic terms in z), and the bottom kernel's data
template <class E>
pb_status mg_build_levels(const E &e, int first, const pb_system *sys, cudaStream_t s) {
    using T = typename E::T;
    const T kap = (T)sys->kap_s;
    for (int l = first; l < e.nlev; ++l) {
        const mg::LevT<T> &C = e.lev[l];
        const unsigned blocks = cdiv((long long)C.nx * C.ny * C.nz, 256);
        if (l == 1 && first == 1)
            k_mg_coarsen<true, T><<<blocks, 256, 0, s>>>(e.lev[0], C, sys->W[0], sys->W[1], sys->W[2], sys->code, kap);
        else if (l > 0)
            k_mg_coarsen<false, T><<<blocks, 256, 0, s>>>(e.lev[l - 1], C, nullptr, nullptr, nullptr, nullptr, (T)0);
        k_mg_diag<<<blocks, 256, 0, s>>>(C);
        note_launch(1);
        PB_LAUNCH_CHECK();
    }
    k_mg_pack<<<cdiv(e.bot, 256), 256, 0, s>>>(e, e.bot);
    PB_LAUNCH_CHECK();
    for (int l = first; l < e.nlev; ++l)  // z held the ionic terms
        PB_CUDA_TRY(cudaMemsetAsync(e.lev[l].z, 0, sizeof(T) * (size_t)e.lev[l].sxy * e.lev[l].nz, s));
    return PB_OK;
}

// the hierarchy of e's levels, in m
pb_status mg_fill(const pb_system *sys, mg::Entry &e, MgState *m, cudaStream_t s) {
    using namespace mg;
    const size_t bytes = mg_layout(e, 1, nullptr);
    m->head = (Head *)dalloc(sizeof(Head), s);
    m->v = (float *)dalloc(sizeof(float) * (size_t)sys->pad.Np, s);
    m->mem = dalloc(bytes, s);
    m->partials = (float *)dalloc(sizeof(float) * e.nu0, s);
    if (!m->head || !m->v || !m->mem || !m->partials) return PB_ERR_OOM;
    PB_CUDA_TRY(cudaMemsetAsync(m->head, 0, sizeof(Head), s));
    PB_CUDA_TRY(cudaMemsetAsync(m->v, 0, sizeof(float) * (size_t)sys->pad.Np, s));
    PB_CUDA_TRY(cudaMemsetAsync(m->mem, 0, bytes, s));
    e.lev[0].s = sys->z32;
    e.lev[0].z = m->v;
    mg_layout(e, 1, (char *)m->mem);
    e.st = sys->st;
    e.cp = make_c32(sys);
    e.dg_in = 6.f * e.cp.w_in;
    e.dg_out = 6.f * e.cp.w_out + e.cp.kap;
    e.partials = m->partials;
    pb_status rc = PB_OK;
    if ((rc = make_map(&e.sd, sys->z32, false, sys->pad, D0W, D0R)) != PB_OK ||
        (rc = make_map(&e.cd, sys->code, true, sys->pad, C0W, D0R)) != PB_OK ||
        (rc = make_map(&e.su, sys->z32, false, sys->pad, U0W, U0R)) != PB_OK ||
        (rc = make_map(&e.cu, sys->code, true, sys->pad, C0W, FY + 1)) != PB_OK)
        return rc;
    if ((rc = mg_build_levels(e, 1, sys, s)) != PB_OK) return rc;
    m->e = e;
    return PB_OK;
}

// A hierarchy that device memory has no room for is done without: Jacobi needs
// none.  The next solve asks again.
pb_status mg_optional(pb_status rc) {
    if (rc != PB_ERR_OOM) return rc;
    set_error("");
    return PB_OK;
}

// hierarchy of a uniform system, built with its first mixed-precision solve
// (coefficients and grids do not change after that); sys->mg is set once all
// of it is there, and stays null on grids without one
pb_status build_mg_state(pb_system *sys, cudaStream_t s) {
    using namespace mg;
    if (sys->mg) return PB_OK;
    Entry e{};
    e.code = sys->code;
    if (!mg_levels(sys->pad, e)) return PB_OK;
    pb_status rc = mg_prepare();
    if (rc != PB_OK) return rc;
    MgState *m = new (std::nothrow) MgState();
    if (!m) return PB_OK;
    if ((rc = mg_fill(sys, e, m, s)) != PB_OK) {
        mg_release(m, s);
        return mg_optional(rc);
    }
    sys->mg = m;
    return PB_OK;
}

template <class K>
unsigned mg_resident(K kernel, int nt) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, nt, 0) != cudaSuccess || per_sm <= 0) {
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

// one V-cycle of one system (z32 -> v, or a lattice's s -> z); returns the
// number of launches
int launch_vcycle(const pb_system *sys, cudaStream_t s) {
    using namespace mg;
    const MgState *m = (const MgState *)sys->mg;
    Entry e = m->e;
    e.st = sys->st;  // the engine lends a system its slot's state
    const bool fine = !m->lattice;
    static const unsigned rd1 = mg_resident(k_mg_down<true>, DNT), ru1 = mg_resident(k_mg_up<true>, UNT);
    const Entry *none = nullptr;
    for (int l = 0; l < e.nbot; ++l) {
        const int n = ditems(e, l);
        if (l == 0 && fine)
            mg_launch(k_mg_down0<true>, n, D0NT, 0, s, true, none, (const Head *)m->head, n, e);
        else
            mg_launch(k_mg_down<true>, std::min<unsigned>(n, rd1), DNT, 0, s, true, none, (const Head *)m->head, l, n, e);
    }
    mg_launch(k_mg_bottom<Entry, true>, 1, BOT_T, mg_bottom_bytes(e), s, true, none, (const Head *)m->head, e);
    for (int l = e.nbot - 1; l >= 0; --l) {
        const int n = uitems(e, l);
        if (l == 0 && fine)
            mg_launch(k_mg_up0<true>, n, U0NT, 0, s, true, none, m->head, n, e);
        else
            mg_launch(k_mg_up<true>, std::min<unsigned>(n, ru1), UNT, 0, s, true, none, (const Head *)m->head, l, n, e);
    }
    return 2 * e.nbot + 1;
}

// the lattice's hierarchy, in m: `up` coarsenings of the lattice that fill() writes
pb_status mg_lattice_fill(const pb_system *sys, mg::Entry &e, int up, lattice_fill fill, MgState *m, cudaStream_t s) {
    using namespace mg;
    m->lattice = true;
    const size_t bytes = mg_layout(e, 0, nullptr);
    m->head = (Head *)dalloc(sizeof(Head), s);
    m->mem = dalloc(bytes, s);
    if (!m->head || !m->mem) return PB_ERR_OOM;
    PB_CUDA_TRY(cudaMemsetAsync(m->head, 0, sizeof(Head), s));
    PB_CUDA_TRY(cudaMemsetAsync(m->mem, 0, bytes, s));
    mg_layout(e, 0, (char *)m->mem);
    e.st = sys->st;
    // from the finest of the lattices down to level 0
    const int n = e.lev[0].nx;
    pb_status rc = PB_OK;
    Lev F{};
    void *tmp = nullptr;
    for (int q = up; q >= 0 && rc == PB_OK; --q) {
        Lev C = e.lev[0];
        void *mem = nullptr;
        if (q > 0) {
            C.nx = C.ny = C.nz = (n - 1) * (1 << q) + 1;
            C.sx = (C.nx + 3) & ~3;
            C.sxy = C.sx * C.ny;
            const size_t c = mg_lev_size(C);
            mem = dalloc(16 * c, s);
            if (!mem) {
                rc = PB_ERR_OOM;
                break;
            }
            C.wx = (float *)mem;
            C.wy = C.wx + c;
            C.wz = C.wy + c;
            C.z = C.wz + c;
            C.dg = nullptr;
        }
        if (q == up) {
            rc = fill(sys, C.nx, C.sx, C.wx, C.wy, C.wz, C.z, s);
        } else {
            k_mg_coarsen<false, float><<<cdiv((long long)C.nx * C.ny * C.nz, 256), 256, 0, s>>>(F, C, nullptr, nullptr,
                                                                                        nullptr, nullptr, 0.f);
            note_launch(1);
        }
        dfree(tmp, s);
        tmp = mem;
        F = C;
    }
    dfree(tmp, s);
    if (rc == PB_OK && cudaGetLastError() != cudaSuccess) rc = PB_ERR_CUDA;
    if (rc == PB_OK) rc = mg_build_levels(e, 0, sys, s);
    m->e = e;
    return rc;
}

// The lattice of an octree's preconditioner, of n nodes an axis; sys->mg stays
// null where memory has no room for it
pb_status mg_lattice_make(pb_system *sys, int n, int up, lattice_fill fill, cudaStream_t s) {
    using namespace mg;
    if (sys->mg) return PB_OK;
    Entry e{};
    PadGeo g{};
    g.nx = g.ny = g.nz = n;
    if (!mg_levels(g, e, true)) return PB_OK;
    pb_status rc = mg_prepare();
    if (rc != PB_OK) return rc;
    MgState *m = new (std::nothrow) MgState();
    if (!m) return PB_OK;
    if ((rc = mg_lattice_fill(sys, e, up, fill, m, s)) != PB_OK) {
        mg_release(m, s);
        return mg_optional(rc);
    }
    sys->mg = m;
    return PB_OK;
}

LatticeMg mg_lattice_view(const pb_system *sys) {
    const mg::Lev &L = ((const MgState *)sys->mg)->e.lev[0];
    LatticeMg v;
    v.n = L.nx;
    v.sx = L.sx;
    v.sxy = L.sxy;
    v.s = L.s;
    v.z = L.z;
    v.dg = L.dg;
    return v;
}

int mg_lattice_cycle(const pb_system *sys, cudaStream_t s) { return launch_vcycle(sys, s); }

// ---- FP64 cycle of the plain FP64 solver
struct Mg64State {
    mg::Entry64 e{};
    double *v = nullptr;  // preconditioned residual (padded)
    void *mem = nullptr;
};

void mg64_release(Mg64State *m, cudaStream_t s) {
    if (!m) return;
    dfree(m->v, s);
    dfree(m->mem, s);
    delete m;
}

void free_mg64_state(pb_system *sys) {
    mg64_release((Mg64State *)sys->mg64, sys->stream);
    sys->mg64 = nullptr;
}

pb_status mg64_fill(const pb_system *sys, mg::Entry64 &e, Mg64State *m, cudaStream_t s) {
    using namespace mg;
    const size_t bytes = mg_layout(e, 1, nullptr), b0 = sizeof(double) * (size_t)sys->pad.Np;
    m->v = (double *)dalloc(b0, s);
    m->mem = dalloc(bytes, s);
    if (!m->v || !m->mem) return PB_ERR_OOM;
    PB_CUDA_TRY(cudaMemsetAsync(m->v, 0, b0, s));
    PB_CUDA_TRY(cudaMemsetAsync(m->mem, 0, bytes, s));
    mg_layout(e, 1, (char *)m->mem);
    LevT<double> &L = e.lev[0];
    L.s = sys->z64;
    L.z = m->v;
    L.wx = sys->op64[0];
    L.wy = sys->op64[1];
    L.wz = sys->op64[2];
    L.dg = sys->op64[3];
    L.di = sys->op64[4];
    L.r = sys->q64;  // q is free between the update and the direction kernels, and zero off the interior
    e.st = sys->st;
    const pb_status rc = mg_build_levels(e, 1, sys, s);
    m->e = e;
    return rc;
}

// built with the first FP64 solve of a uniform system; sys->mg64 is set once
// all of it is there, and stays null on grids without a hierarchy
pb_status build_mg64_state(pb_system *sys, cudaStream_t s) {
    using namespace mg;
    if (sys->mg64) return PB_OK;
    Entry64 e{};
    if (!mg_levels(sys->pad, e)) return PB_OK;
    pb_status rc = mg_prepare();
    if (rc != PB_OK) return rc;
    Mg64State *m = new (std::nothrow) Mg64State();
    if (!m) return PB_OK;
    if ((rc = mg64_fill(sys, e, m, s)) != PB_OK) {
        mg64_release(m, s);
        return mg_optional(rc);
    }
    sys->mg64 = m;
    return PB_OK;
}

// one FP64 V-cycle (z64 -> v); returns the number of launches
int launch_vcycle64(const pb_system *sys, cudaStream_t s) {
    using namespace mg;
    const Entry64 &e = ((const Mg64State *)sys->mg64)->e;
    auto blocks = [](const LevT<double> &L) {
        return cdiv((long long)(L.nx - 2) * (L.ny - 2) * (L.nz - 2), 256);
    };
    for (int l = 0; l < e.nbot; ++l) {
        mg_launch(k_mg64_residual, blocks(e.lev[l]), 256, 0, s, true, e.lev[l], (const CgState *)sys->st);
        mg_launch(k_mg64_restrict, blocks(e.lev[l + 1]), 256, 0, s, true, e.lev[l], e.lev[l + 1],
                  (const CgState *)sys->st);
    }
    mg_launch(k_mg_bottom<Entry64, true>, 1, BOT_T, mg_bottom_bytes(e), s, true, (const Entry64 *)nullptr,
              (const Head *)nullptr, e);
    static const unsigned top = mg_resident(k_mg64_smooth<true>, 256);
    for (int l = e.nbot - 1; l >= 0; --l) {
        mg_launch(k_mg64_correct, blocks(e.lev[l]), 256, 0, s, true, e.lev[l], e.lev[l + 1], (const CgState *)sys->st);
        if (l == 0)
            mg_launch(k_mg64_smooth<true>, std::min(blocks(e.lev[l]), top), 256, 0, s, true, e.lev[l], sys->st,
                      sys->partials);
        else
            mg_launch(k_mg64_smooth<false>, blocks(e.lev[l]), 256, 0, s, true, e.lev[l], sys->st, (double *)nullptr);
    }
    return 4 * e.nbot + 1;
}
