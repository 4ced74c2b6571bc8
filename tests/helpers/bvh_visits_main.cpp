// Node visits and triangle tests of rays through the BVH2: the exact boxes against the kernels' 32-byte
// records (DevBVH2, walked link by link with their grids).  One line per scene:
//   name, triangles, grids, then per ray: exact nodes, record nodes, exact triangles, record triangles
// Arguments: triangles of a detailed object (about), rays per scene.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "cr_internal.h"

using V = std::vector<float>;
struct Ray {
    double o[3], d[3];
};

static uint64_t state = 1;
static double urand() {
    state = state * 6364136223846793005ull + 1442695040888963407ull;
    return (double)(state >> 11) * 0x1.0p-53;
}

static void tri(V& v, const double* a, const double* b, const double* c) {
    for (const double* p : {a, b, c})
        for (int k = 0; k < 3; ++k) v.push_back((float)p[k]);
}

// a sphere of n x 2n quads
static void sphere(V& v, double cx, double cy, double cz, double r, int n) {
    auto at = [&](int i, int j, double* p) {
        const double th = M_PI * i / n, ph = M_PI * j / n;
        p[0] = cx + r * std::sin(th) * std::cos(ph);
        p[1] = cy + r * std::cos(th);
        p[2] = cz + r * std::sin(th) * std::sin(ph);
    };
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < 2 * n; ++j) {
            double a[3], b[3], c[3], d[3];
            at(i, j, a);
            at(i + 1, j, b);
            at(i + 1, j + 1, c);
            at(i, j + 1, d);
            tri(v, a, b, c);
            tri(v, a, c, d);
        }
}

// a plane of half extent h at height y, m x m quads
static void ground(V& v, double y, double h, int m) {
    for (int i = 0; i < m; ++i)
        for (int j = 0; j < m; ++j) {
            const double x0 = -h + 2 * h * i / m, x1 = -h + 2 * h * (i + 1) / m, z0 = -h + 2 * h * j / m,
                         z1 = -h + 2 * h * (j + 1) / m;
            const double a[3] = {x0, y, z0}, b[3] = {x1, y, z0}, c[3] = {x1, y, z1}, d[3] = {x0, y, z1};
            tri(v, a, b, c);
            tri(v, a, c, d);
        }
}

static bool hit_tri(const float* p, const Ray& r, double& t) { // Moeller-Trumbore
    double e1[3], e2[3], s[3];
    for (int k = 0; k < 3; ++k) {
        e1[k] = (double)p[3 + k] - p[k];
        e2[k] = (double)p[6 + k] - p[k];
        s[k] = r.o[k] - p[k];
    }
    auto cross = [](const double* a, const double* b, double* c) {
        c[0] = a[1] * b[2] - a[2] * b[1];
        c[1] = a[2] * b[0] - a[0] * b[2];
        c[2] = a[0] * b[1] - a[1] * b[0];
    };
    auto dot = [](const double* a, const double* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; };
    double q[3], w[3];
    cross(r.d, e2, q);
    const double det = dot(e1, q);
    if (det == 0) return false;
    const double u = dot(s, q) / det;
    cross(s, e1, w);
    const double x = dot(r.d, w) / det, tt = dot(e2, w) / det;
    if (u < 0 || x < 0 || u + x > 1 || !(tt > 0) || !(tt < t)) return false;
    t = tt;
    return true;
}

// entry distance of a box, +inf when missed or behind t
static double enter(const Ray& r, const double* lo, const double* hi, double t) {
    double a = 0, b = t;
    for (int k = 0; k < 3; ++k) {
        if (r.d[k] == 0) {
            if (r.o[k] < lo[k] || r.o[k] > hi[k]) return INFINITY;
            continue;
        }
        double x = (lo[k] - r.o[k]) / r.d[k], y = (hi[k] - r.o[k]) / r.d[k];
        if (x > y) std::swap(x, y);
        a = std::max(a, x);
        b = std::min(b, y);
    }
    return a <= b ? a : INFINITY;
}

struct Walk {
    const V& v;
    const cr::HostBVH2& b;
    const cr::DevBVH2& d;
    bool exact;
    uint64_t nodes = 0, tris = 0;
    double t = 0;

    double plane(uint32_t in, uint32_t q, int k) const { // back in the scene's units
        float f, lo = d.lo[k], scale = d.scale[k];
        const uint32_t bits = 0x3f000000u | q << 8;
        std::memcpy(&f, &bits, 4);
        if (in) {
            std::memcpy(&lo, &d.words[8 * (size_t)in + k], 4);
            std::memcpy(&scale, &d.words[8 * (size_t)in + 3 + k], 4);
        }
        return ((double)f - 0.5) / scale + lo;
    }
    void leaf(uint32_t code, const Ray& r) {
        for (uint32_t i = code >> 2; i <= (code >> 2) + (code & 3u); ++i) {
            ++tris;
            hit_tri(&v[9 * (size_t)b.leaf_order[i]], r, t);
        }
    }
    void node(uint32_t i, uint32_t in, const Ray& r) { // in: the way in to its grid, 0 the scene's
        ++nodes;
        double lo[2][3], hi[2][3], at[2];
        uint32_t link[2];
        const uint32_t* rec = &d.words[8 * (size_t)i];
        const float* o = &b.nodes[16 * (size_t)i];
        static const int lower[3][2] = {{0, 4}, {2, 6}, {8, 10}};
        for (int w = 0; w < 2; ++w) {
            for (int k = 0; k < 3; ++k) {
                const uint32_t q = rec[3 * w + k];
                lo[w][k] = exact ? o[lower[k][w]] : plane(in, q & 0xffffu, k);
                hi[w][k] = exact ? o[lower[k][w] + 1] : plane(in, q >> 16, k);
            }
            std::memcpy(&link[w], exact ? (const void*)&o[12 + w] : &rec[6 + w], 4);
            at[w] = enter(r, lo[w], hi[w], t);
        }
        const int first = at[0] <= at[1] ? 0 : 1;
        for (int w : {first, 1 - first}) {
            if (at[w] == INFINITY || at[w] > t) continue;
            if ((int32_t)link[w] >= 0) {
                node(link[w], in, r);
            } else if (~link[w] & cr::kGridLink) {
                const uint32_t g = ~link[w] & ~cr::kGridLink;
                node(d.words[8 * (size_t)g + 7], g, r);
            } else {
                leaf(~link[w], r);
            }
        }
    }
};

static void scene(const char* name, const V& v, const std::vector<Ray>& rays) {
    const uint32_t n = (uint32_t)(v.size() / 9);
    const cr::HostBVH2 b = cr::build_bvh2(v.data(), n, 8);
    const cr::DevBVH2 d = cr::pack_bvh2(b, 8);
    Walk e{v, b, d, true}, q{v, b, d, false};
    for (const Ray& r : rays) {
        e.t = q.t = INFINITY;
        e.node(0, 0, r);
        q.node(0, 0, r);
        if (e.t != q.t) {
            std::printf("%s: a ray hits at %.17g through the exact boxes, at %.17g through the records\n", name, e.t, q.t);
            std::exit(1);
        }
    }
    const double m = (double)rays.size();
    std::printf("%s %u %u %.2f %.2f %.2f %.2f\n", name, n, d.n_grids, e.nodes / m, q.nodes / m, e.tris / m, q.tris / m);
}

// rays from distance `far` at points around a centre
static std::vector<Ray> rays_at(double cx, double cy, double cz, double far, int n) {
    std::vector<Ray> out;
    while ((int)out.size() < n) {
        Ray r;
        double len = 0;
        for (int k = 0; k < 3; ++k) {
            r.o[k] = 2 * urand() - 1;
            len += r.o[k] * r.o[k];
        }
        if (len > 1 || len < 1e-4) continue;
        const double c[3] = {cx, cy, cz};
        for (int k = 0; k < 3; ++k) {
            r.o[k] = c[k] + far * r.o[k] / std::sqrt(len);
            r.d[k] = c[k] + 1.6 * urand() - 0.8 - r.o[k];
        }
        r.o[1] = c[1] + std::fabs(r.o[1] - c[1]);
        out.push_back(r);
    }
    return out;
}

int main(int argc, char** argv) {
    const int n_obj = argc > 1 ? std::atoi(argv[1]) : 100000, n_rays = argc > 2 ? std::atoi(argv[2]) : 500;
    const int n = std::max(4, (int)std::sqrt(n_obj / 4.0));
    for (double half : {5.0, 50.0, 500.0, 5000.0, 50000.0, 5e6}) {
        V v;
        sphere(v, 0, 0, 0, 1, n);
        ground(v, -1, half, 1);
        scene(("ground" + std::to_string((long)half)).c_str(), v, rays_at(0, 0, 0, 3, n_rays));
    }
    { // ground of many quads
        V v;
        sphere(v, 0, 0, 0, 1, n);
        ground(v, -1, 5000, 100);
        scene("tiled", v, rays_at(0, 0, 0, 3, n_rays));
    }
    { // many objects a kilometre apart, away from the origin
        V v;
        std::vector<Ray> rays;
        for (int i = 0; i < 8; ++i)
            for (int j = 0; j < 8; ++j) {
                sphere(v, 1000.0 * i, 0, 1000.0 * j, 1, std::max(4, n / 8));
                const auto r = rays_at(1000.0 * i, 0, 1000.0 * j, 3, std::max(1, n_rays / 64));
                rays.insert(rays.end(), r.begin(), r.end());
            }
        ground(v, -1, 10000, 16);
        scene("town", v, rays);
    }
    { // detail within detail: a sphere on a table in a house in a country
        V v;
        sphere(v, 0, 0, 0, 0.001, n / 2);
        for (double h : {0.01, 1.0, 100.0, 10000.0, 1e6}) ground(v, -0.001 - 0.1 * h, h, 24);
        std::vector<Ray> rays = rays_at(0, 0, 0, 3, n_rays);
        for (Ray& r : rays)
            for (int k = 0; k < 3; ++k) {
                r.o[k] *= 0.001;
                r.d[k] *= 0.001;
            }
        scene("nested", v, rays);
    }
    { // even detail: one grid is enough
        V v;
        sphere(v, 0, 0, 0, 1, n);
        scene("even", v, rays_at(0, 0, 0, 3, n_rays));
    }
    return 0;
}
