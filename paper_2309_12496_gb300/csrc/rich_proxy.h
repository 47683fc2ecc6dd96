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

// The crossings of one ray with one proxy. cell >= 0: the cell to look up at
// distance t; -1: the ray cannot meet the mesh there. sure: the margins hold
// for this ray; if not, the BVH has to take it. t_max: the nearest hit known so far;
// (dx, dy, dz) a unit vector to 1e-6, |o| at most the scene's o_max.
//
// The bounds: with u = 2^-24 and W >= |o - c|, the FP32 crossing point differs
// from the ray's exact crossing of the sphere or plane by at most 8 u W across
// the surface (the roundings of w, of the dots and, after the Newton step on
// |p| = r, of |p|^2 - r^2), by 8 u W / c along the ray for an angle of
// incidence with cosine c >= kProxyCosMin, and a facet's point lies within
// `shell` of the surface. The cells' margin, which is also DevProxy::dt, holds the
// longest way of such a ray through shell + E, E = 32 u W, and E once more: for a
// plane (shell + E) / kProxyCosMin + E, for a sphere somewhat more, as a ray that
// enters it flattens (shell_reach in rich_proxy.cpp). A crossing is found by selects instead of branches: a
// warp's rays mostly take the same surfaces, and control flow was a fifth of the
// trace's instructions.
constexpr float kProxyCosMin = 0.25f;

#ifdef __CUDA_ARCH__
RICH_HD float proxy_div(float a, float b) { return __fdividef(a, b); }
RICH_HD float proxy_rsqrt(float a) { return rsqrtf(a); }
#else
RICH_HD float proxy_div(float a, float b) { return a / b; }
RICH_HD float proxy_rsqrt(float a) { return 1.0f / sqrtf(a); }
#endif

// Whether the ray passes by the sphere that bounds the proxy's mesh, or meets it
// beyond t_max or behind the start only. (|w|^2 - (w . d)^2 is off by at most
// 16 u W^2, which g2 holds.)
RICH_HD bool proxy_misses(const DevProxy &P, float ox, float oy, float oz, float dx, float dy,
                          float dz, float t_max) {
    const float wx = ox - P.gx, wy = oy - P.gy, wz = oz - P.gz;
    const float w2 = fmaf(wx, wx, fmaf(wy, wy, wz * wz));
    const float tb = -fmaf(wx, dx, fmaf(wy, dy, wz * dz));
    return (fmaf(-tb, tb, w2) > P.g2) | ((tb < 0.0f) & (w2 > P.g2)) | (tb - P.g_r > t_max);
}

// The cell of the point p (relative to c) at distance t, or -1.
RICH_HD int proxy_cell(const DevProxy &P, float px, float py, float pz, float t, float t_min,
                       float t_max, bool ok) {
    const float x = fmaf(px, P.e1x, fmaf(py, P.e1y, fmaf(pz, P.e1z, -P.x0)));
    const float y = fmaf(px, P.e2x, fmaf(py, P.e2y, fmaf(pz, P.e2z, -P.y0)));
    ok = ok & (x >= 0.0f) & (x < P.fnx) & (y >= 0.0f) & (y < P.fny) & (t >= t_min - P.dt) &
         (t <= t_max + P.dt);
    return ok ? P.first_cell + (int)y * P.nx + (int)x : -1;
}

RICH_HD int proxy_plane(const DevProxy &P, float ox, float oy, float oz, float dx, float dy,
                        float dz, float t_min, float t_max, float &t, bool &sure) {
    const float wx = ox - P.cx, wy = oy - P.cy, wz = oz - P.cz;
    const float den = fmaf(dx, P.ax, fmaf(dy, P.ay, dz * P.az));
    t = -proxy_div(fmaf(wx, P.ax, fmaf(wy, P.ay, wz * P.az)), den);
    sure = fabsf(den) >= kProxyCosMin;
    return proxy_cell(P, fmaf(t, dx, wx), fmaf(t, dy, wy), fmaf(t, dz, wz), t, t_min, t_max, sure);
}

// A sphere's crossing on leaving it (side = 1) or entering it (side = -1), from
// b = w . d and h2 = r^2 - |w - b d|^2 >= h2_min.
RICH_HD int proxy_sphere_side(const DevProxy &P, float wx, float wy, float wz, float dx, float dy,
                              float dz, float b, float h2, float side, float t_min, float t_max,
                              float &t, bool ok) {
    const float ih = side * proxy_rsqrt(h2);
    t = fmaf(h2, ih, -b);
    float px = fmaf(t, dx, wx), py = fmaf(t, dy, wy), pz = fmaf(t, dz, wz);
    // one Newton step on |p|^2 = r^2 (d|p|^2/dt = +-2 h at the crossings)
    const float s = -0.5f * ih * fmaf(px, px, fmaf(py, py, fmaf(pz, pz, -P.r2)));
    t += s;
    px = fmaf(s, dx, px);
    py = fmaf(s, dy, py);
    pz = fmaf(s, dz, pz);
    ok = ok & (fmaf(px, P.ax, fmaf(py, P.ay, pz * P.az)) >= P.z_min);
    return proxy_cell(P, px, py, pz, t, t_min, t_max, ok);
}

// The sphere's crossing on leaving; entering: whether the crossing on entering
// may lie ahead too (proxy_sphere_side with side = -1 then finds its cell).
RICH_HD int proxy_sphere(const DevProxy &P, float ox, float oy, float oz, float dx, float dy,
                         float dz, float t_min, float t_max, float &t, bool &sure, bool &entering,
                         float &b, float &h2) {
    const float wx = ox - P.cx, wy = oy - P.cy, wz = oz - P.cz;
    b = fmaf(wx, dx, fmaf(wy, dy, wz * dz));
    const float qx = fmaf(-b, dx, wx), qy = fmaf(-b, dy, wy), qz = fmaf(-b, dz, wz);
    const float q2 = fmaf(qx, qx, fmaf(qy, qy, qz * qz));
    h2 = P.r2 - q2;
    const bool meets = h2 >= P.h2_min;
    sure = meets | (q2 > P.q2_max);
    h2 = meets ? h2 : P.h2_min;
    // -b - h >= t_far (behind the start whatever the roundings if below)
    const float far = -b - P.t_far;
    entering = meets & (far >= 0.0f) & (far * far >= h2);
    return proxy_sphere_side(P, wx, wy, wz, dx, dy, dz, b, h2, 1.0f, t_min, t_max, t, meets);
}

// The cells that a ray has to look up: of its two nearest crossings that have one
// (c0, c1, at t0 <= t1; -1: none), and the distance of a third (infinity: none).
struct ProxyCells {
    int c0, c1;
    float t0, t1, t2;
    bool sure;             // the margins hold for the ray at every proxy
};

// S: n_proxies and proxies(), the planes first. skip_px: the proxy code of the
// triangle just left, or 0. Its proxy is passed over when that is its only surface;
// when its surfaces lie apart, its entry crossing (the start) lists none but the
// one left (RICH1, 10^4 tracks, 482 -> 457 us; RICH2 3.76 -> 3.54 ms).
template <class Proxies>
RICH_HD ProxyCells proxy_cells(const Proxies &S, int n_planes, float ox, float oy, float oz,
                               float dx, float dy, float dz, uint32_t skip_px, float t_min,
                               float t_max) {
    const float kInf = HUGE_VALF;
    ProxyCells r{-1, -1, kInf, kInf, kInf, true};
    auto keep = [&](float t, int c) {
        t = c >= 0 ? t : kInf;
        const bool l0 = t < r.t0, l1 = t < r.t1;
        r.t2 = fminf(r.t2, l1 ? r.t1 : t);
        r.c1 = l0 ? r.c0 : (l1 ? c : r.c1);
        r.t1 = l0 ? r.t0 : (l1 ? t : r.t1);
        r.c0 = l0 ? c : r.c0;
        r.t0 = l0 ? t : r.t0;
    };
    unsigned entering = 0;
    const int left = (int)(skip_px & kProxyIndex) - 1;
    const int own = skip_px & kProxySingle ? left : -1;
    const unsigned no_entry = skip_px & kProxyApart ? 1u << left : 0u;
#pragma unroll 1
    for (int i = 0; i < S.n_proxies; ++i) {
        const DevProxy &P = S.proxies()[i];
        if (proxy_misses(P, ox, oy, oz, dx, dy, dz, t_max) | (i == own)) continue;
        float t;
        bool sure;
        int c;
        if (i < n_planes) {
            c = proxy_plane(P, ox, oy, oz, dx, dy, dz, t_min, t_max, t, sure);
        } else {
            float sb, h2;
            bool ent;
            c = proxy_sphere(P, ox, oy, oz, dx, dy, dz, t_min, t_max, t, sure, ent, sb, h2);
            entering |= (unsigned)ent << i;
        }
        r.sure = r.sure & sure;
        keep(t, c);
    }
    entering &= ~no_entry;
    while (entering) {
#ifdef __CUDA_ARCH__
        const DevProxy &P = S.proxies()[__ffs(entering) - 1];
#else
        const DevProxy &P = S.proxies()[__builtin_ctz(entering)];
#endif
        entering &= entering - 1u;
        const float wx = ox - P.cx, wy = oy - P.cy, wz = oz - P.cz;
        const float sb = fmaf(wx, dx, fmaf(wy, dy, wz * dz));
        const float qx = fmaf(-sb, dx, wx), qy = fmaf(-sb, dy, wy), qz = fmaf(-sb, dz, wz);
        const float h2 = P.r2 - fmaf(qx, qx, fmaf(qy, qy, qz * qz));
        float t;
        const int c = proxy_sphere_side(P, wx, wy, wz, dx, dy, dz, sb, h2, -1.0f, t_min, t_max, t,
                                        true);
        keep(t, c);
    }
    return r;
}

// Host builder. On return `proxies` is empty when some triangle fits no
// proxy (the scene then uses the BVH alone).
struct ProxyResult {
    std::vector<DevProxy> proxies;
    std::vector<std::vector<DevProxyCell>> cells;   // one grid per proxy, in order
    std::vector<int32_t> lists;       // triangle lists of the cells with more than two
    std::vector<int32_t> list_cells;  // (while building) those cells
    std::vector<uint32_t> tri_code;   // proxy code of every triangle
    int n_planes = 0;                 // planes first, then spheres
    float o2_max = 0.0f;              // |o|^2 up to which the bounds hold
    float dt_max = 0.0f;              // largest dt of any proxy
};

// tris: in leaf order, DevTri::pad naming the triangle's surface; extent:
// largest absolute coordinate of the scene.
void build_proxies(const std::vector<DevTri> &tris, double extent, ProxyResult &out);

}  // namespace rich
