// Re-triangulated molecular surface for the first integral of Eq.
// energy_ion (Sec. 3.3.2): the surface is rebuilt cell by cell by marching
// cubes whose vertices are the analytic intersection points r_p of the
// crossing edges (end nodes in different media), with the analytic normal of
// the ball surface at each vertex; the integral then takes the vertex rule
// T_j/3 on every triangle, with phi at the vertices from Eq. phi0 (in the
// energy kernel).
//
// One cell's triangles, without a case table: on each face the crossing
// edges are joined in pairs (two crossings: one segment; four, the ambiguous
// face: two segments that each cut off one inside corner, so both cells of a
// face agree and the surface is closed).  Every crossing edge of the cell
// lies on two faces, so the segments close into loops; a loop starts at its
// lowest cell-edge index, first goes to the smaller of that vertex's two
// neighbours, and is cut into the fan (v0, v_m, v_m+1).
//
// k_mc_weight gives every crossing point W = sum of T_j/3 over the triangles
// of its (up to four) cells that have it as a vertex, visiting the cells in
// node order and their triangles in fan order, so each sum is formed in one
// fixed order without atomics.  k_mc_normal finds, through the atom cell
// list, the ball whose sphere passes closest to the point (smallest
// | |r_p - c| - R |, ties to the lower atom index) and takes the unit vector
// from its centre; an FP32 pass first bounds that minimum, so that the FP64
// comparison only visits the candidates that can reach it.  This file is compiled without FMA contraction, so every
// value is reproducible to the bit.
#include <math.h>

#include "pb_internal.h"

namespace pbg {

namespace {

// cell corners: bit 0 = +x, bit 1 = +y, bit 2 = +z.  Cell edges: 0-3 along
// x, 4-7 along y, 8-11 along z (corner pairs below).
constexpr int EDGE_CORNER[12][2] = {{0, 1}, {2, 3}, {4, 5}, {6, 7}, {0, 2}, {1, 3},
                                    {4, 6}, {5, 7}, {0, 4}, {1, 5}, {2, 6}, {3, 7}};
// faces: corners in cyclic order, and the cell edge between corner q and q+1
constexpr int FACE[6][4] = {{0, 2, 6, 4}, {1, 3, 7, 5}, {0, 1, 5, 4}, {2, 3, 7, 6}, {0, 1, 3, 2}, {4, 5, 7, 6}};
constexpr int FACE_EDGE[6][4] = {{4, 10, 6, 8}, {5, 11, 7, 9}, {0, 9, 2, 8}, {1, 11, 3, 10}, {0, 5, 1, 4}, {2, 7, 3, 6}};

// The triangles of a cell depend on its corner flags alone, so the
// construction above runs once for each of the 256 patterns, in the compiler:
// t[0] triangles in fan order, each as three 4-bit cell edges.
struct CellTriangles {
    uint16_t t[256][16];
};
constexpr CellTriangles make_triangles() {
    CellTriangles out{};
    for (int ins = 0; ins < 256; ++ins) {
        int nb[12][2] = {}, has[12] = {};
        bool crossed[12] = {}, seen[12] = {};
        for (int e = 0; e < 12; ++e)
            crossed[e] = (((ins >> EDGE_CORNER[e][0]) ^ (ins >> EDGE_CORNER[e][1])) & 1) != 0;
        for (int f = 0; f < 6; ++f) {
            int cr[4] = {}, m = 0;
            for (int q = 0; q < 4; ++q)
                if (((ins >> FACE[f][q]) ^ (ins >> FACE[f][(q + 1) & 3])) & 1) cr[m++] = q;
            int pair[2][2] = {}, pairs = 0;
            if (m == 2) {
                pair[0][0] = FACE_EDGE[f][cr[0]];
                pair[0][1] = FACE_EDGE[f][cr[1]];
                pairs = 1;
            } else if (m == 4) {
                // cut off each inside corner (corner q lies between face edges q-1 and q)
                const int q0 = ((ins >> FACE[f][0]) & 1) ? 0 : 1;
                pair[0][0] = FACE_EDGE[f][(q0 + 3) & 3];
                pair[0][1] = FACE_EDGE[f][q0];
                pair[1][0] = FACE_EDGE[f][(q0 + 1) & 3];
                pair[1][1] = FACE_EDGE[f][(q0 + 2) & 3];
                pairs = 2;
            }
            for (int p = 0; p < pairs; ++p)
                for (int e = 0; e < 2; ++e) {
                    const int a = pair[p][e];
                    nb[a][has[a]++] = pair[p][1 - e];
                }
        }
        int count = 0;
        for (int e0 = 0; e0 < 12; ++e0) {
            if (!crossed[e0] || seen[e0]) continue;
            int loop[12] = {e0}, len = 1, prev = e0;
            int cur = nb[e0][0] < nb[e0][1] ? nb[e0][0] : nb[e0][1];
            seen[e0] = true;
            while (cur != e0 && len < 12) {
                loop[len++] = cur;
                seen[cur] = true;
                const int nx = nb[cur][0] == prev ? nb[cur][1] : nb[cur][0];
                prev = cur;
                cur = nx;
            }
            for (int m = 1; m + 1 < len; ++m)
                out.t[ins][1 + count++] = (uint16_t)(loop[0] | loop[m] << 4 | loop[m + 1] << 8);
        }
        out.t[ins][0] = (uint16_t)count;
    }
    return out;
}
__device__ const CellTriangles d_triangles = make_triangles();

// place of edge id in the crossing list (-1 if absent)
__device__ __forceinline__ int find_edge(const uint16_t *__restrict__ emask, const int *__restrict__ epos,
                                         long long id) {
    const unsigned m = emask[id >> 4], b = (unsigned)id & 15u;
    if (!((m >> b) & 1u)) return -1;
    return epos[id >> 4] + __popc(m & ((1u << b) - 1u));
}

__global__ void __launch_bounds__(128)
k_mc_weight(GridGeo g, const uint8_t *__restrict__ inside, const long long *__restrict__ ids,
            const uint16_t *__restrict__ emask, const int *__restrict__ epos, const int8_t *__restrict__ sign,
            const double *__restrict__ rp, long long ncross, double *__restrict__ W) {
    const long long s = blockIdx.x * 128ll + threadIdx.x;
    const bool on = s < ncross && sign[s] != 0;
    const long long sy = g.nx, sz = (long long)g.nx * g.ny;
    int d = 0, i = 0, j = 0, k = 0;
    if (on) {
        const long long id = ids[s];
        d = (int)(id / g.N);
        const long long a = id - (long long)d * g.N, r = a / g.nx;
        i = (int)(a - r * g.nx);
        k = (int)(r / g.ny);
        j = (int)(r - (long long)k * g.ny);
    }
    // The walk over the triangles that have the point as a vertex: the (up to
    // four) cells around the edge in node order, each cell's triangles in fan
    // order.  The edge's index in a cell: x edges 0-3 by (dy + 2 dz), y
    // edges 4-7 by (dx + 2 dz), z edges 8-11 by (dx + 2 dy), offsets from the
    // cell.  FP64 instructions cost a warp the same for one lane as for all, so
    // every lane walks to its next triangle before the warp measures them
    // (257^3, 580,000 points: each cell triangulated anew with binary searches for its
    // points 1,870 us, the triangle table and direct look-ups 630 us, this
    // order 307 us).
    int cell = on ? -1 : 4, q = 0, count = 0, es = 0;
    const uint16_t *tri = nullptr;
    long long n0 = 0;
    auto next = [&]() -> unsigned {
        for (;;) {
            while (q >= count) {
                if (++cell >= 4) {
                    cell = 4;
                    return ~0u;
                }
                const int u = cell & 1, v = cell >> 1;
                const int ci = d == 0 ? i : i - 1 + u, cj = d == 0 ? j - 1 + u : (d == 1 ? j : j - 1 + v),
                          ck = d == 2 ? k : k - 1 + v;
                q = count = 0;
                if (ci < 0 || cj < 0 || ck < 0 || ci > g.nx - 2 || cj > g.ny - 2 || ck > g.nz - 2) continue;
                const int ox = i - ci, oy = j - cj, oz = k - ck;
                es = d == 0 ? oy + 2 * oz : (d == 1 ? 4 + ox + 2 * oz : 8 + ox + 2 * oy);
                n0 = ((long long)ck * g.ny + cj) * g.nx + ci;
                unsigned ins = 0;
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    ins |= (inside[n0 + (c & 1) + ((c >> 1) & 1) * sy + ((c >> 2) & 1) * sz] ? 1u : 0u) << c;
                tri = d_triangles.t[ins];
                count = tri[0];
            }
            const unsigned t = tri[1 + q++];
            if ((int)(t & 15u) == es || (int)((t >> 4) & 15u) == es || (int)(t >> 8) == es) return t;
        }
    };
    double w = 0.0;
    for (;;) {
        const unsigned t = next();
        __syncwarp();
        if (!__any_sync(0xffffffffu, t != ~0u)) break;
        if (t != ~0u) {
            double p[3][3];
            bool ok = true;
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                long long at = s;
                const int e = (int)((t >> (4 * v)) & 15u);
                if (e != es) {
                    // the edge's low corner: x edges (0, dy, dz), y edges (dx, 0, dz), z edges (dx, dy, 0)
                    const int ax = e >> 2, u = e & 1, z = (e >> 1) & 1;
                    const long long low = n0 + (ax == 0 ? u * sy + z * sz : (ax == 1 ? u + z * sz : u + z * sy));
                    at = find_edge(emask, epos, (long long)ax * g.N + low);
                    ok = ok && at >= 0;
                }
                at = ok ? at : s;
                p[v][0] = rp[3 * at];
                p[v][1] = rp[3 * at + 1];
                p[v][2] = rp[3 * at + 2];
            }
            if (ok) {
                const double u0 = p[1][0] - p[0][0], u1 = p[1][1] - p[0][1], u2 = p[1][2] - p[0][2];
                const double v0 = p[2][0] - p[0][0], v1 = p[2][1] - p[0][1], v2 = p[2][2] - p[0][2];
                const double x = u1 * v2 - u2 * v1;
                const double y = u2 * v0 - u0 * v2;
                const double z = u0 * v1 - u1 * v0;
                // T/3 correctly rounded without a division: with c = RN(1/3) the
                // product's remainder is exact in one fused multiply-add
                const double area = 0.5 * sqrt((x * x + y * y) + z * z), c = 1.0 / 3.0, third = area * c;
                w += fma(fma(-3.0, third, area), c, third);
            }
        }
        __syncwarp();
    }
    if (s < ncross) W[s] = w;
}

// |r - c| - R in FP32 differs from the FP64 value by at most about
// 4 * 2^-24 * X, X the largest coordinate relative to the cell list's corner
// (each rounding of a coordinate to FP32 costs 2^-24 X, the difference and
// the distance add rounding of their own); a candidate whose FP32 value
// exceeds the FP32 minimum by more than twice that bound can be neither the
// FP64 minimum nor tied with it.  The cell list's margin is several times that.

__global__ void __launch_bounds__(128)
k_mc_normal(CellList cl, const int8_t *__restrict__ sign, const double *__restrict__ rp, long long ncross,
            double *__restrict__ nrm) {
    const long long s = blockIdx.x * 128ll + threadIdx.x;
    if (s >= ncross) return;
    double o0 = 0.0, o1 = 0.0, o2 = 0.0;
    if (sign[s] != 0) {
        const double p0 = rp[3 * s], p1 = rp[3 * s + 1], p2 = rp[3 * s + 2];
        const double p[3] = {p0, p1, p2};
        int cc[3];
        for (int q = 0; q < 3; ++q) {
            const double u = floor((p[q] - cl.lo[q]) / cl.cs);
            cc[q] = (u < -4.0) ? -4 : ((u > (double)cl.dim[q] + 4.0) ? cl.dim[q] + 4 : (int)u);
        }
        const float f0 = (float)(p0 - cl.lo[0]), f1 = (float)(p1 - cl.lo[1]),
                    f2 = (float)(p2 - cl.lo[2]);
        const int cx0 = max(cc[0] - 1, 0), cx1 = min(cc[0] + 1, cl.dim[0] - 1);
        // the atoms of the 27 cells, a run for every row of cells
        auto scan = [&](auto f) {
            if (cx0 > cx1) return;
            for (int row = 0; row < 9; ++row) {
                const int cy = cc[1] - 1 + row % 3, cz = cc[2] - 1 + row / 3;
                if (cz < 0 || cz >= cl.dim[2] || cy < 0 || cy >= cl.dim[1]) continue;
                const int c0 = (cz * cl.dim[1] + cy) * cl.dim[0];
                for (int q = cl.start[c0 + cx0], q1 = cl.start[c0 + cx1 + 1]; q < q1; ++q) {
                    const float4 a = cl.a32[q];
                    const float dx = f0 - a.x, dy = f1 - a.y, dz = f2 - a.z;
                    f(q, fabsf(sqrtf(dx * dx + dy * dy + dz * dz) - a.w));
                }
            }
        };
        // pass 1: the smallest FP32 deviation
        float m32 = INFINITY;
        scan([&](int, float dev) { m32 = fminf(m32, dev); });
        // pass 2: the FP64 comparison over the candidates that can win, noted
        // first and then evaluated by the warp together (one or two a point)
        const float lim = m32 + cl.margin;
        int best = -1, bat = -1;
        double bdev = 0.0, bd = 0.0;
        auto compare = [&](int q) {
            const double4 a = cl.a64[q];
            const int at = cl.atom[q];
            const double dx = p0 - a.x, dy = p1 - a.y, dz = p2 - a.z;
            const double dd = sqrt((dx * dx + dy * dy) + dz * dz);
            const double dev = fabs(dd - a.w);
            if (best < 0 || dev < bdev || (dev == bdev && at < bat)) {
                best = q;
                bat = at;
                bdev = dev;
                bd = dd;
            }
        };
        int n = 0, c0 = 0, c1 = 0, c2 = 0, c3 = 0;
        scan([&](int q, float dev32) {
            if (dev32 > lim) return;
            if (n == 0) c0 = q;
            else if (n == 1) c1 = q;
            else if (n == 2) c2 = q;
            else if (n == 3) c3 = q;
            else compare(q);
            ++n;
        });
        __syncwarp(__activemask());
        if (n > 0) compare(c0);
        if (n > 1) compare(c1);
        if (n > 2) compare(c2);
        if (n > 3) compare(c3);
        if (best >= 0) {
            const double4 a = cl.a64[best];
            o0 = (p0 - a.x) / bd;
            o1 = (p1 - a.y) / bd;
            o2 = (p2 - a.z) / bd;
        }
    }
    nrm[3 * s] = o0;
    nrm[3 * s + 1] = o1;
    nrm[3 * s + 2] = o2;
}

}  // namespace

// Vertex weights and normals of the re-triangulated surface, from the
// uniform grid pass (the grid itself, or an octree's finest lattice).
pb_status mc_surface(pb_grid *g, const uint16_t *emask, const int *epos, cudaStream_t s) {
    const long long nc = g->ncross;
    g->mc_w = (double *)dalloc(sizeof(double) * (size_t)(nc > 0 ? nc : 1), s);
    g->mc_n = (double *)dalloc(sizeof(double) * 3 * (size_t)(nc > 0 ? nc : 1), s);
    if (!g->mc_w || !g->mc_n) return PB_ERR_OOM;
    if (nc == 0) return PB_OK;
    k_mc_weight<<<cdiv(nc, 128), 128, 0, s>>>(g->geo, g->inside, g->cid, emask, epos, g->csign, g->crp, nc, g->mc_w);
    PB_LAUNCH_CHECK();
    k_mc_normal<<<cdiv(nc, 128), 128, 0, s>>>(g->cells, g->csign, g->crp, nc, g->mc_n);
    PB_LAUNCH_CHECK();
    return PB_OK;
}

}  // namespace pbg
