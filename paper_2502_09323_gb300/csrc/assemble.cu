// Coefficient assembly and right-hand side.
//
// Compiled with --fmad=false so the FP64 coefficients and the charge deposit
// are reproducible to the bit (each expression evaluated as written).
//
// Sec. 3.1: with vertex quadrature the Nedelec mass matrix is diagonal and
//   static condensation leaves the 7-point operator A = G^T W G + C, W_e the
//   edge weight eps_e h, C_kk = eps_s k_D^2 h^3 at solvent nodes (the ionic
//   term c = eps_s k_D^2 chi_s of Sec. 2.1 lumped on the node).
// Sec. 3.2 (Eq. WHA): 1/eps_e = alpha/eps_m + (1 - alpha)/eps_s.
// Eq. RVop: f_k = R(w_k) = sum_i q_i w_k(r_i), times 4 pi l_B in reduced units,
//   plus W_e phi_b for every edge that reaches a Dirichlet node.
#include <math.h>

#include "pb_internal.h"

namespace pbg {

namespace {

// Row (j, k) of a thread's node and its first index; one warp takes a row at
// a time, so that no node needs a division.
struct Row {
    int j, k;
    long long a;  // canonical index of node (0, j, k)
};
__device__ __forceinline__ Row row_of(const GridGeo &g, long long r) {
    Row w;
    w.k = (int)(r / g.ny);
    w.j = (int)(r - (long long)w.k * g.ny);
    w.a = r * g.nx;
    return w;
}
constexpr int ROWS = 8;  // rows (warps) of a block

// Pure-medium weights for every existing edge; the code byte of the padded
// FP32 layout starts as the solute bit.
__global__ void __launch_bounds__(32 * ROWS)
k_coef_pure(const uint8_t *__restrict__ inside, GridGeo g, PadGeo p, double w_in, double w_out,
            double *__restrict__ Wx, double *__restrict__ Wy, double *__restrict__ Wz, uint8_t *__restrict__ code) {
    const long long r = blockIdx.x * (long long)ROWS + threadIdx.y;
    if (r >= (long long)g.ny * g.nz) return;
    const Row w = row_of(g, r);
    for (int i = threadIdx.x; i < g.nx; i += 32) {
        const int in = inside[w.a + i];
        const double v = in ? w_in : w_out;
        Wx[w.a + i] = (i < g.nx - 1) ? v : 0.0;
        Wy[w.a + i] = (w.j < g.ny - 1) ? v : 0.0;
        Wz[w.a + i] = (w.k < g.nz - 1) ? v : 0.0;
        code[r * p.sx + i] = (uint8_t)in;
    }
}

// Listed edges: WHA weight; FP32 copy for the compressed operator; flag bit
// (1 + d) of the low node's code byte.
__global__ void k_coef_special(const long long *__restrict__ ids, const double *__restrict__ alpha,
                               long long ncross, GridGeo g, PadGeo p, double eps_in,
                               double eps_out, double *__restrict__ Wx, double *__restrict__ Wy,
                               double *__restrict__ Wz, float *__restrict__ wx32,
                               float *__restrict__ wy32, float *__restrict__ wz32,
                               uint8_t *__restrict__ code) {
    long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (s >= ncross) return;
    long long e = ids[s];
    int d = (int)(e / g.N);
    long long a = e - (long long)d * g.N;
    double al = alpha[s];
    double w = 1.0 / (al / eps_in + (1.0 - al) / eps_out) * g.h;
    double *W = d == 0 ? Wx : (d == 1 ? Wy : Wz);
    W[a] = w;
    long long i = a % g.nx, j = (a / g.nx) % g.ny, k = a / ((long long)g.nx * g.ny);
    long long pa = (k * g.ny + j) * p.sx + i;
    float *w32 = d == 0 ? wx32 : (d == 1 ? wy32 : wz32);
    w32[pa] = (float)w;
    unsigned int *word = (unsigned int *)(code + (pa & ~3ll));
    atomicOr(word, (unsigned int)(2u << d) << (8 * (pa & 3)));
}

// diag = ((((((Wx- + Wx+) + Wy-) + Wy+) + Wz-) + Wz+) + kappa), 0 on boundary.
// An unlisted edge joins two nodes of one medium and has its pure weight, so a
// node whose six edges are unlisted (its code bytes say so) has one of two
// diagonals, formed by the same additions on the host: seven FP64 additions
// a node had bound this kernel (257^3 228 us).
__global__ void __launch_bounds__(32 * ROWS)
k_diag(const double *__restrict__ Wx, const double *__restrict__ Wy, const double *__restrict__ Wz,
       const uint8_t *__restrict__ code, GridGeo g, PadGeo p, double kap_s, double d_in, double d_out,
       double *__restrict__ diag) {
    const long long r = blockIdx.x * (long long)ROWS + threadIdx.y;
    if (r >= (long long)g.ny * g.nz) return;
    const Row w = row_of(g, r);
    const bool rim = w.j == 0 || w.k == 0 || w.j == g.ny - 1 || w.k == g.nz - 1;
    const long long sy = g.nx, sz = (long long)g.nx * g.ny;
    for (int i = threadIdx.x; i < g.nx; i += 32) {
        const long long a = w.a + i;
        double s = 0.0;
        if (!rim && i > 0 && i < g.nx - 1) {
            const uint8_t *c = code + r * p.sx + i;
            if (((c[0] & 0xE) | (c[-1] & 2) | (c[-p.sx] & 4) | (c[-p.sxy] & 8)) == 0) {
                s = (c[0] & 1) ? d_in : d_out;
            } else {
                s = s + Wx[a - 1];
                s = s + Wx[a];
                s = s + Wy[a - sy];
                s = s + Wy[a];
                s = s + Wz[a - sz];
                s = s + Wz[a];
                s = s + ((c[0] & 1) ? 0.0 : kap_s);
            }
        }
        diag[a] = s;
    }
}

__global__ void k_kappa(const uint8_t *__restrict__ inside, long long N, double kap_s,
                        double *__restrict__ out) {
    long long a = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (a < N) out[a] = inside[a] ? 0.0 : kap_s;
}

// Trilinear cell and weights of atom j (cell = clamp(floor((x-o)/h), 0, n-2)).
struct Tri {
    long long c[3];
    double w[3][2];
};

__device__ __forceinline__ Tri tri_cell(const GridGeo &g, double x, double y, double z) {
    Tri t;
    double p[3] = {x, y, z};
    long long nn[3] = {g.nx, g.ny, g.nz};
    for (int d = 0; d < 3; ++d) {
        double u = (p[d] - g.o[d]) / g.h;
        long long c = (long long)floor(u);
        c = c < 0 ? 0 : (c > nn[d] - 2 ? nn[d] - 2 : c);
        double tt = u - (double)c;
        t.c[d] = c;
        t.w[d][0] = 1.0 - tt;
        t.w[d][1] = tt;
    }
    return t;
}

// One thread per (atom, corner).  The contributions to a node are summed in
// increasing atom order, starting from 0, by the thread of the smallest atom
// id touching that node -- the same order as a sequential loop over atoms, so
// the result is deterministic and independent of scheduling.
__global__ void k_deposit(const double *__restrict__ atoms, long long na, GridGeo g,
                          CellList cl, const int *__restrict__ cstart,
                          const int *__restrict__ clist, double coef0,
                          double *__restrict__ f) {
    long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= 8 * na) return;
    long long i = t >> 3;
    int corner = (int)(t & 7);
    const double *X = atoms, *Y = atoms + na, *Z = atoms + 2 * na, *Q = atoms + 4 * na;
    Tri ti = tri_cell(g, X[i], Y[i], Z[i]);
    long long node[3] = {ti.c[0] + (corner & 1), ti.c[1] + ((corner >> 1) & 1),
                         ti.c[2] + ((corner >> 2) & 1)};
    // position of the node, cell of the node in the atom cell list
    double xa[3];
    float x32[3];
    int cc[3];
    for (int d = 0; d < 3; ++d) {
        xa[d] = g.o[d] + (double)node[d] * g.h;
        x32[d] = (float)(xa[d] - cl.lo[d]);
        double u = floor((xa[d] - cl.lo[d]) / cl.cs);
        cc[d] = (u < -4.0) ? -4 : ((u > (double)cl.dim[d] + 4.0) ? cl.dim[d] + 4 : (int)u);
    }
    // an atom whose cell has the node as a corner lies within h of it along
    // every axis; FP32 (with the cell list's margin) passes the others over
    const float reach = (float)(1.0001 * g.h) + cl.margin;
    const int cx0 = max(cc[0] - 1, 0), cx1 = min(cc[0] + 1, cl.dim[0] - 1);
    // atoms whose cell has this node as a corner, in id order, MAXC at a time
    // (one round unless more than MAXC charges share the node)
    constexpr int MAXC = 32;
    int ids[MAXC], last = -1;
    double acc = 0.0;
    for (;;) {
        int m = 0;
        for (int cz = cc[2] - 1; cz <= cc[2] + 1; ++cz) {
            if (cz < 0 || cz >= cl.dim[2] || cx0 > cx1) continue;
            for (int cy = cc[1] - 1; cy <= cc[1] + 1; ++cy) {
                if (cy < 0 || cy >= cl.dim[1]) continue;
                const int c0 = (cz * cl.dim[1] + cy) * cl.dim[0];
                for (int s = cstart[c0 + cx0], s1 = cstart[c0 + cx1 + 1]; s < s1; ++s) {
                    const float4 b = cl.a32[s];
                    if (fabsf(b.x - x32[0]) > reach || fabsf(b.y - x32[1]) > reach || fabsf(b.z - x32[2]) > reach)
                        continue;
                    const int j = clist[s];
                    if (j <= last || (m == MAXC && j > ids[MAXC - 1])) continue;
                    const Tri tj = (j == i) ? ti : tri_cell(g, X[j], Y[j], Z[j]);
                    bool corner_of = true;
                    for (int d = 0; d < 3; ++d) {
                        long long off = node[d] - tj.c[d];
                        if (off != 0 && off != 1) corner_of = false;
                    }
                    if (!corner_of) continue;
                    int q = m < MAXC ? m++ : MAXC - 1;  // a full list drops its largest id
                    while (q > 0 && ids[q - 1] > j) {
                        ids[q] = ids[q - 1];
                        --q;
                    }
                    ids[q] = j;
                }
            }
        }
        if (last < 0 && (m == 0 || ids[0] != (int)i)) return;  // another thread owns this node
        for (int q = 0; q < m; ++q) {
            int j = ids[q];
            Tri tj = (j == i) ? ti : tri_cell(g, X[j], Y[j], Z[j]);
            int dx = (int)(node[0] - tj.c[0]), dy = (int)(node[1] - tj.c[1]),
                dz = (int)(node[2] - tj.c[2]);
            double coef = coef0 * Q[j];
            acc += coef * (tj.w[0][dx] * tj.w[1][dy] * tj.w[2][dz]);
        }
        if (m < MAXC) break;
        last = ids[MAXC - 1];
    }
    f[(node[2] * g.ny + node[1]) * g.nx + node[0]] = acc;
}

// f[a] += W_e phi_b for edges to Dirichlet nodes, in the order -x,+x,-y,+y,-z,+z.
// Only nodes next to the boundary have such edges: a warp takes a row, whole
// rows in the outer layers and the two end nodes of the others.
__global__ void __launch_bounds__(32 * ROWS)
k_lift(const double *__restrict__ Wx, const double *__restrict__ Wy, const double *__restrict__ Wz,
       const double *__restrict__ bc, GridGeo g, double *__restrict__ f) {
    const long long r = blockIdx.x * (long long)ROWS + threadIdx.y;
    if (r >= (long long)g.ny * g.nz) return;
    const Row w = row_of(g, r);
    const int j = w.j, k = w.k;
    if (j == 0 || k == 0 || j == g.ny - 1 || k == g.nz - 1) return;
    const bool layer = j == 1 || k == 1 || j == g.ny - 2 || k == g.nz - 2;
    const double *W[3] = {Wx, Wy, Wz};
    const long long st[3] = {1, g.nx, (long long)g.nx * g.ny};
    const int n[3] = {g.nx, g.ny, g.nz};
    const int count = layer ? g.nx - 2 : (g.nx > 3 ? 2 : 1);
    for (int q = threadIdx.x; q < count; q += 32) {
        const int i = layer ? 1 + q : (q ? g.nx - 2 : 1);
        const long long a = w.a + i;
        const int c[3] = {i, j, k};
        double v = f[a];
        for (int d = 0; d < 3; ++d) {
            if (c[d] - 1 == 0) v += W[d][a - st[d]] * bc[a - st[d]];
            if (c[d] + 1 == n[d] - 1) v += W[d][a] * bc[a + st[d]];
        }
        f[a] = v;
    }
}

}  // namespace

pb_status assemble(pb_system *sys, cudaStream_t s) {
    pb_grid *g = sys->g;
    const GridGeo &geo = g->geo;
    const long long N = geo.N;
    PadGeo &p = sys->pad;
    p.nx = geo.nx;
    p.ny = geo.ny;
    p.nz = geo.nz;
    p.sx = (geo.nx + 15) & ~15;  // 16 elements: TMA strides and code rows need 16 B
    p.sxy = (long long)p.sx * geo.ny;
    p.Np = p.sxy * geo.nz;
    p.N = N;
    for (int d = 0; d < 3; ++d) sys->W[d] = (double *)dalloc(sizeof(double) * N, s);
    sys->diag = (double *)dalloc(sizeof(double) * N, s);
    sys->rhs = (double *)dalloc(sizeof(double) * N, s);
    sys->bc = (double *)dalloc(sizeof(double) * N, s);
    sys->phi = (double *)dalloc(sizeof(double) * N, s);
    sys->code = (uint8_t *)dalloc((size_t)((p.Np + 15) & ~15ll), s);
    for (int d = 0; d < 3; ++d) sys->w32[d] = (float *)dalloc(sizeof(float) * p.Np, s);
    if (!sys->W[0] || !sys->W[1] || !sys->W[2] || !sys->diag || !sys->rhs || !sys->bc ||
        !sys->phi || !sys->code || !sys->w32[0] || !sys->w32[1] || !sys->w32[2])
        return PB_ERR_OOM;
    PB_CUDA_TRY(cudaMemsetAsync(sys->code, 0, (size_t)((p.Np + 15) & ~15ll), s));
    PB_CUDA_TRY(cudaMemsetAsync(sys->bc, 0, sizeof(double) * N, s));
    const double eps_in = sys->p.eps_in, eps_out = sys->p.eps_out, h = geo.h;
    const dim3 rows(32, ROWS);
    const unsigned rblocks = cdiv((long long)geo.ny * geo.nz, ROWS);
    k_coef_pure<<<rblocks, rows, 0, s>>>(g->inside, geo, p, eps_in * h, eps_out * h, sys->W[0], sys->W[1], sys->W[2],
                                         sys->code);
    PB_LAUNCH_CHECK();
    if (g->ncross > 0) {
        k_coef_special<<<cdiv(g->ncross, 256), 256, 0, s>>>(g->cid, g->calpha, g->ncross, geo, p,
                                                            eps_in, eps_out, sys->W[0], sys->W[1],
                                                            sys->W[2], sys->w32[0], sys->w32[1],
                                                            sys->w32[2], sys->code);
        PB_LAUNCH_CHECK();
    }
    // diagonals of a node with six pure edges, added as k_diag adds them
    auto pure = [](double w, double kap) {
        volatile double t = 0.0;
        for (int q = 0; q < 6; ++q) t = t + w;
        return (double)(t + kap);
    };
    k_diag<<<rblocks, rows, 0, s>>>(sys->W[0], sys->W[1], sys->W[2], sys->code, geo, p, sys->kap_s,
                                    pure(eps_in * h, 0.0), pure(eps_out * h, sys->kap_s), sys->diag);
    PB_LAUNCH_CHECK();
    return PB_OK;
}

pb_status deposit_rhs(pb_system *sys, cudaStream_t s) {
    pb_grid *g = sys->g;
    const GridGeo &geo = g->geo;
    PB_CUDA_TRY(cudaMemsetAsync(sys->rhs, 0, sizeof(double) * geo.N, s));
    double coef0 = 4.0 * M_PI * sys->lB;
    if (g->na > 0) {
        k_deposit<<<cdiv(8 * g->na, 128), 128, 0, s>>>(g->atoms, g->na, geo, g->cells,
                                                       g->cells.start, g->cells.atom, coef0,
                                                       sys->rhs);
        PB_LAUNCH_CHECK();
    }
    if (sys->p.bc != PB_BC_ZERO) {  // zero boundary values lift nothing
        k_lift<<<cdiv((long long)geo.ny * geo.nz, ROWS), dim3(32, ROWS), 0, s>>>(sys->W[0], sys->W[1], sys->W[2],
                                                                               sys->bc, geo, sys->rhs);
        PB_LAUNCH_CHECK();
    }
    return PB_OK;
}

pb_status fill_kappa(const pb_system *sys, double *dst, cudaStream_t s) {
    k_kappa<<<cdiv(sys->g->geo.N, 256), 256, 0, s>>>(sys->g->inside, sys->g->geo.N, sys->kap_s,
                                                     dst);
    PB_LAUNCH_CHECK();
    return PB_OK;
}

}  // namespace pbg
