// rich_proxy.h -- surface proxies: where a ray can meet a meshed mirror.
//
// A mesh of a spherical or flat mirror lies in a thin shell around one sphere
// or plane (its vertices on it, its facets at most the sagitta inside). A
// ray's hit on that sphere or plane then says, to a fraction of a
// millimetre, which facets it can meet: the mesh is projected along the
// proxy's axis onto a grid whose cells list the triangles within a margin of
// the cell, and a ray tests the triangles of one cell in place of walking
// the BVH. The triangles themselves are tested as the BVH's leaves are, so
// the nearest hit is the same; a ray for which the margin does not hold
// (grazing, far away, or a direction that is not a unit vector) is reported
// and takes the BVH.
#pragma once

#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "rich_internal.h"

#ifdef __CUDACC__
#define RICH_HD __host__ __device__ __forceinline__
#else
#define RICH_HD inline
#endif

namespace rich {

// One proxy against a ray: cell[k] >= 0 is the cell to test at the ray's
// k-th crossing (two for a sphere, nearer first), -1 none. Returns false when
// the ray may meet the mesh but the margin does not hold (take the BVH).
// t_max: the nearest hit known so far; (dx, dy, dz) a unit vector to 1e-6.
//
// The bounds: with u = 2^-24 and W = sqrt(w2_max) >= |o - c|, the FP32
// crossing point differs from the ray's exact crossing of the sphere or
// plane by at most 8 u W across the surface (the roundings of w, of the
// dots and, after the Newton step on |p| = r, of |p|^2 - r^2), by 8 u W / c
// along the ray for an angle of incidence with cosine c >= kProxyCosMin,
// and a facet's point lies within `shell` of the surface; the cells' margin
// holds (shell + E) / kProxyCosMin + E with E = 32 u W.
constexpr float kProxyCosMin = 0.25f;

RICH_HD bool proxy_cells(const DevProxy &P, float ox, float oy, float oz, float dx, float dy,
                         float dz, float t_min, float t_max, int cell[2]) {
    cell[0] = cell[1] = -1;
    const float wx = ox - P.cx, wy = oy - P.cy, wz = oz - P.cz;
    const float w2 = fmaf(wx, wx, fmaf(wy, wy, wz * wz));
    bool sure = w2 <= P.w2_max;
    const float b = fmaf(wx, dx, fmaf(wy, dy, wz * dz));
    float t[2];
    int n = 1;
    float half_inv_h = 0.0f;
    if (P.r > 0.0f) {
        const float qx = fmaf(-b, dx, wx), qy = fmaf(-b, dy, wy), qz = fmaf(-b, dz, wz);
        const float q2 = fmaf(qx, qx, fmaf(qy, qy, qz * qz));
        if (sure && q2 > P.q2_max) return true;                  // passes outside the shell
        const float h2 = P.r2 - q2;
        sure = sure && h2 >= P.h2_min;
        if (sure) {
            const float h = sqrtf(h2);
            half_inv_h = 0.5f / h;
            t[0] = -b - h;
            t[1] = -b + h;
            n = 2;
        }
    } else {
        const float den = fmaf(dx, P.ax, fmaf(dy, P.ay, dz * P.az));
        sure = sure && fabsf(den) >= kProxyCosMin;
        if (sure) t[0] = -fmaf(wx, P.ax, fmaf(wy, P.ay, wz * P.az)) / den;
    }
    if (!sure) {
        // may the ray meet the sphere that bounds the mesh?
        const float gx = wx - P.gx, gy = wy - P.gy, gz = wz - P.gz;
        const float gb = fmaf(gx, dx, fmaf(gy, dy, gz * dz));
        const float mx = fmaf(-gb, dx, gx), my = fmaf(-gb, dy, gy), mz = fmaf(-gb, dz, gz);
        const float m2 = fmaf(mx, mx, fmaf(my, my, mz * mz));
        return w2 <= P.w2_max && m2 > P.g2;
    }
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 0; k < 2; ++k) {
        if (k >= n) continue;
        float tk = t[k];
        if (tk < P.t_far) continue;      // behind the start whatever the roundings
        float px = fmaf(tk, dx, wx), py = fmaf(tk, dy, wy), pz = fmaf(tk, dz, wz);
        if (P.r > 0.0f) {
            // one Newton step on |p|^2 = r^2 (d|p|^2/dt = -+2h at the roots)
            const float f = fmaf(px, px, fmaf(py, py, fmaf(pz, pz, -P.r2)));
            const float s = k == 0 ? f * half_inv_h : -f * half_inv_h;
            tk += s;
            px = fmaf(s, dx, px);
            py = fmaf(s, dy, py);
            pz = fmaf(s, dz, pz);
            if (!(fmaf(px, P.ax, fmaf(py, P.ay, pz * P.az)) >= P.z_min)) continue;
        }
        if (tk < t_min - P.dt || tk > t_max + P.dt) continue;
        const float x = (fmaf(px, P.e1x, fmaf(py, P.e1y, pz * P.e1z)) - P.x0) * P.inv_cell;
        const float y = (fmaf(px, P.e2x, fmaf(py, P.e2y, pz * P.e2z)) - P.y0) * P.inv_cell;
        if (!(x >= 0.0f && x < P.fnx && y >= 0.0f && y < P.fny)) continue;
        cell[k] = P.first_cell + (int)y * P.nx + (int)x;
    }
    return true;
}

// Host builder. On return `proxies` is empty when some triangle fits no
// proxy (the scene then uses the BVH alone).
struct ProxyResult {
    std::vector<DevProxy> proxies;
    std::vector<DevProxyCell> cells;
    std::vector<int32_t> lists;       // triangle lists of the cells with more than two
};

// tris: in leaf order, DevTri::pad naming the triangle's surface; extent:
// largest absolute coordinate of the scene.
void build_proxies(const std::vector<DevTri> &tris, double extent, ProxyResult &out);

}  // namespace rich
