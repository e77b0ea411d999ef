// The plane structure of a leaf (2D) or block (3D) and its face coefficients,
// shared by the leaf kernels and the host's plan of their storage.
//
// A leaf is a stack of H planes of nb cells (2D: rows of w cells; 3D: x-y
// planes of w_x w_y cells), eliminated from both ends towards plane M = H / 2
// (kernels_leaf.cu).  The columns of B (one per segment) that have met a
// plane when it is eliminated from below (h = 0) are, in this order: the
// segments of the low side (y- / z-), the lateral patches that span all
// planes (3D), then per group of G planes, from the lowest, one run of
// segments per lateral side; from above (h = 1) likewise from the high side
// and the highest group down.  So a plane's columns are a prefix of its
// half's order.
#pragma once
#include "mrcm_internal.h"

namespace mrcm {

struct LeafGeo {
    int nb, H, m, M, w0;          // cells per plane, planes, segments, middle plane, cells per plane row
    int G, ngr, nf, ncoarse;      // planes per lateral group, groups, segments per group, spanning patches
    int end_off[2], n_end[2];     // first segment and number of segments of the low / high side
    int lat_off[4], lat_w[4];     // lateral sides: first segment; segments per group (0: absent, -1: one
                                  // patch over all planes)
    long long L_off, Z_off, zb_off, R_off, r_off;

    __host__ __device__ int halfplanes(int h) const { return h ? H - 1 - M : M; }
    // columns that have met plane k of half h
    __host__ __device__ int cols(int h, int k) const {
        return n_end[h] + ncoarse + (h ? ngr - k / G : k / G + 1) * nf;
    }
    __host__ __device__ int ncols(int h) const { return halfplanes(h) > 0 ? cols(h, h ? M + 1 : M - 1) : 0; }
    // the segment of column p of half h
    __host__ __device__ int segment(int h, int p) const {
        if (p < n_end[h]) return end_off[h] + p;
        p -= n_end[h];
        if (p < ncoarse) {
            for (int s = 0; s < 4; ++s)
                if (lat_w[s] < 0 && p-- == 0) return lat_off[s];
        }
        p -= ncoarse;
        const int r = p / nf, grp = h ? ngr - 1 - r : r;
        p -= r * nf;
        for (int s = 0; s < 4; ++s) {
            if (lat_w[s] <= 0) continue;
            if (p < lat_w[s]) return lat_off[s] + grp * lat_w[s] + p;
            p -= lat_w[s];
        }
        return 0;
    }
    // sum of k' / G + 1 over k' < k
    __host__ __device__ int groups_below(int k) const {
        const int a = k / G, b = k % G;
        return G * a * (a + 1) / 2 + b * (a + 1);
    }
    __host__ __device__ int cols_below(int k) const { return k * (n_end[0] + ncoarse) + nf * groups_below(k); }
    __host__ __device__ int cols_above(int k) const {       // planes k + 1 .. H - 1, from above
        const int c = H - 1 - k;
        return c * (n_end[1] + ncoarse) + nf * (c * (ngr + 1) - (groups_below(H) - groups_below(k + 1)));
    }
    // offset of the stored Z of plane k (h = 0: planes up to M, h = 1: above)
    __host__ __device__ int zoff(int h, int k) const {
        return nb * (h ? cols_below(M) + m + cols_above(k) : cols_below(k));
    }
    __host__ __device__ int zsize() const { return nb * (cols_below(M) + m + cols_above(M)); }
};

__host__ __device__ inline LeafGeo leaf_geo2(const LeafDesc& L, int gx, int gy) {
    LeafGeo g;
    g.nb = L.w; g.H = L.h; g.m = L.m; g.M = L.h / 2; g.w0 = L.w;
    g.G = gy; g.ngr = (L.h + gy - 1) / gy; g.ncoarse = 0;
    g.nf = 0;
    for (int s = 0; s < 4; ++s) { g.lat_off[s] = 0; g.lat_w[s] = 0; }
    for (int s = 0; s < 2; ++s) {
        g.lat_off[s] = L.side_off[s];
        g.lat_w[s] = L.side_off[s] >= 0 ? 1 : 0;
        g.nf += g.lat_w[s];
        g.end_off[s] = L.side_off[2 + s];
        g.n_end[s] = L.side_off[2 + s] >= 0 ? (L.w + gx - 1) / gx : 0;
    }
    g.L_off = L.L_off; g.Z_off = L.Z_off; g.zb_off = L.zb_off; g.R_off = L.R_off; g.r_off = L.r_off;
    return g;
}
__host__ __device__ inline LeafGeo leaf_geo3(const LeafDesc3& B) {
    LeafGeo g;
    g.nb = B.w[0] * B.w[1]; g.H = B.w[2]; g.m = B.m; g.M = B.w[2] / 2; g.w0 = B.w[0];
    g.G = 1; g.ngr = B.w[2]; g.nf = g.ncoarse = 0;
    for (int s = 0; s < 4; ++s) {
        g.lat_off[s] = B.side_off[s];
        g.lat_w[s] = B.side_off[s] < 0 ? 0 : (B.side_fine[s] ? (s < 2 ? B.w[1] : B.w[0]) : -1);
        if (g.lat_w[s] > 0) g.nf += g.lat_w[s];
        if (g.lat_w[s] < 0) ++g.ncoarse;
    }
    for (int s = 0; s < 2; ++s) {
        g.end_off[s] = B.side_off[4 + s];
        g.n_end[s] = B.side_off[4 + s] < 0 ? 0 : (B.side_fine[4 + s] ? g.nb : 1);
    }
    g.L_off = B.L_off; g.Z_off = B.Z_off; g.zb_off = B.zb_off; g.R_off = B.R_off; g.r_off = B.r_off;
    return g;
}

#ifdef __CUDACC__
namespace {

__device__ __forceinline__ long long cell3(const Grid3& G, int i, int j, int k) {
    return ((long long)k * G.ny + j) * G.nx + i;
}
__device__ __forceinline__ long long xface3(const Grid3& G, int i, int j, int k) {
    return ((long long)k * G.ny + j) * (G.nx + 1) + i;
}
__device__ __forceinline__ long long yface3(const Grid3& G, int i, int j, int k) {
    return ((long long)k * (G.ny + 1) + j) * G.nx + i;
}
__device__ __forceinline__ long long zface3(const Grid3& G, int i, int j, int k) {
    return ((long long)k * G.ny + j) * G.nx + i;
}
__device__ __forceinline__ double area3(const Grid3& G, int d) {
    return d == 0 ? G.hy * G.hz : (d == 1 ? G.hx * G.hz : G.hx * G.hy);
}
// Boundary value of the face of global cell (gi, gj, gk) on domain side s.
__device__ __forceinline__ double bc_value3(const Grid3& G, const double* bc_val, int s, int gi, int gj, int gk) {
    const long long sx = (long long)G.ny * G.nz, sy = (long long)G.nx * G.nz, sz = (long long)G.nx * G.ny;
    long long o;
    if (s < 2) o = (s ? sx : 0) + (long long)gk * G.ny + gj;
    else if (s < 4) o = 2 * sx + (s == 3 ? sy : 0) + (long long)gk * G.nx + gi;
    else o = 2 * sx + 2 * sy + (s == 5 ? sz : 0) + (long long)gj * G.nx + gi;
    return bc_val[o];
}

template <int DIM>
__device__ __forceinline__ LeafGeo leaf_geo(const DevView& v, int leaf) {
    if constexpr (DIM == 2) return leaf_geo2(v.leaves[leaf], v.gx, v.gy);
    else return leaf_geo3(v.leaves3[leaf]);
}

// Cell i of plane k of a leaf: its position and the coefficients of its
// faces seen from it, in the order x-, x+, y-, y+ (, z-, z+).
template <int DIM>
struct CellFaces {
    int x, y, z;               // global cell
    long long cell;
    double c[2 * DIM];
    __device__ __forceinline__ double diag() const {
        if constexpr (DIM == 2) return (c[0] + c[1]) + (c[2] + c[3]);
        else return ((((c[0] + c[1]) + c[2]) + c[3]) + c[4]) + c[5];
    }
    // towards the plane below / above, and to the cell before in the plane
    __device__ __forceinline__ double down() const { return c[2 * DIM - 2]; }
    __device__ __forceinline__ double up() const { return c[2 * DIM - 1]; }
};
template <int DIM>
__device__ __forceinline__ CellFaces<DIM> cell_faces(const DevView& v, int leaf, const LeafGeo& g, int k, int i) {
    CellFaces<DIM> f;
    if constexpr (DIM == 2) {
        const LeafDesc& L = v.leaves[leaf];
        const GridDesc& G = v.grids[L.grid];
        f.x = L.i0 + i; f.y = L.j0 + k; f.z = 0;
        f.cell = G.c0 + (long long)f.y * G.nx + f.x;
        const long long fx = G.fx0 + f.x + (long long)(G.nx + 1) * f.y;
        const long long fy = G.fy0 + f.x + (long long)G.nx * f.y;
        f.c[0] = v.cxU[fx];
        f.c[1] = v.cxL[fx + 1];
        f.c[2] = v.cyU[fy];
        f.c[3] = v.cyL[fy + G.nx];
    } else {
        const LeafDesc3& L = v.leaves3[leaf];
        const Grid3& G = v.g3;
        f.x = L.i0 + i % g.w0; f.y = L.j0 + i / g.w0; f.z = L.k0 + k;
        f.cell = cell3(G, f.x, f.y, f.z);
        f.c[0] = v.cxU[xface3(G, f.x, f.y, f.z)];
        f.c[1] = v.cxL[xface3(G, f.x + 1, f.y, f.z)];
        f.c[2] = v.cyU[yface3(G, f.x, f.y, f.z)];
        f.c[3] = v.cyL[yface3(G, f.x, f.y + 1, f.z)];
        f.c[4] = v.czU[zface3(G, f.x, f.y, f.z)];
        f.c[5] = v.czL[zface3(G, f.x, f.y, f.z + 1)];
    }
    return f;
}
// fn(segment, side) for every skeleton face of cell i of plane k
template <int DIM, class Fn>
__device__ __forceinline__ void skeleton_faces(const LeafGeo& g, int k, int i, Fn&& fn) {
    const int ix = i % g.w0, iy = i / g.w0, w1 = g.nb / g.w0;
    auto lateral = [&](int s, int u) {
        fn(g.lat_off[s] + (g.lat_w[s] > 0 ? (k / g.G) * g.lat_w[s] + u : 0), s);
    };
    if (g.lat_w[0] && ix == 0) lateral(0, DIM == 3 ? iy : 0);
    if (g.lat_w[1] && ix == g.w0 - 1) lateral(1, DIM == 3 ? iy : 0);
    if (DIM == 3 && g.lat_w[2] && iy == 0) lateral(2, ix);
    if (DIM == 3 && g.lat_w[3] && iy == w1 - 1) lateral(3, ix);
}
// the segment of cell i on the low (h = 0) or high (h = 1) side, -1 when the
// side is on the domain boundary; gx: faces per segment there (2D)
template <int DIM>
__device__ __forceinline__ int end_segment(const DevView& v, const LeafGeo& g, int h, int i) {
    if (g.n_end[h] == 0) return -1;
    if (DIM == 2) return g.end_off[h] + i / v.gx;
    return g.end_off[h] + (g.n_end[h] > 1 || g.nb == 1 ? i : 0);
}
// fn(segment, rho) for every skeleton face of the cell
template <int DIM, class Fn>
__device__ __forceinline__ void plane_faces(const DevView& v, const LeafGeo& g, const CellFaces<DIM>& f, int k, int i,
                                            Fn&& fn) {
    skeleton_faces<DIM>(g, k, i, [&](int t, int s) { fn(t, f.c[s]); });
    if (k == 0 && g.n_end[0]) fn(end_segment<DIM>(v, g, 0, i), f.down());
    if (k == g.H - 1 && g.n_end[1]) fn(end_segment<DIM>(v, g, 1, i), f.up());
}

// Sum of rho over the faces of local segment t seen from the leaf's cells, in
// a fixed order (planes outer, cells of the plane inner).
template <int DIM>
__device__ double segment_rho_sum(const DevView& v, int leaf, const LeafGeo& g, int t) {
    double sum = 0.0;
    int k0 = 0, k1 = g.H;
    for (int h = 0; h < 2; ++h)
        if (g.n_end[h] && t >= g.end_off[h] && t < g.end_off[h] + g.n_end[h]) {
            const int k = h ? g.H - 1 : 0;
            for (int i = 0; i < g.nb; ++i)
                if (end_segment<DIM>(v, g, h, i) == t) {
                    const CellFaces<DIM> f = cell_faces<DIM>(v, leaf, g, k, i);
                    sum += h ? f.up() : f.down();
                }
            return sum;
        }
    // a lateral segment: its group of planes (a spanning patch: every plane)
    for (int s = 0; s < 4; ++s) {
        const int w = g.lat_w[s];
        if (w == 0 || t < g.lat_off[s] || t >= g.lat_off[s] + (w > 0 ? w * g.ngr : 1)) continue;
        if (w > 0) {
            k0 = (t - g.lat_off[s]) / w * g.G;
            k1 = min(k0 + g.G, g.H);
        }
        const int w1 = g.nb / g.w0;
        for (int k = k0; k < k1; ++k)
            for (int u = 0; u < (s < 2 ? w1 : g.w0); ++u) {
                if (w > 0 && DIM == 3 && u != (t - g.lat_off[s]) % w) continue;
                const int i = s < 2 ? u * g.w0 + (s ? g.w0 - 1 : 0) : (s == 2 ? 0 : w1 - 1) * g.w0 + u;
                sum += cell_faces<DIM>(v, leaf, g, k, i).c[s];
            }
        return sum;
    }
    return sum;
}

}  // namespace
#endif
}  // namespace mrcm
