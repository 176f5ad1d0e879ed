// gs_delaunay.cu -- Delaunay triangulation of tracked pixels (paper Sec.
// III-A: the image is divided into triangles with the tracked pixels as
// vertices, and points in flat regions take the mean depth of their
// triangle's vertices).  Host code: the triangulation is built on the CPU
// while the GPU selects the pixels and interpolates (gs_pointcloud.cu).
//
// Bowyer-Watson insertion with exact predicates on integer coordinates
// (orientation in 64-bit, in-circle in 64- or 128-bit integers) and "ghost"
// triangles for the outside: every hull edge (a, b) carries a triangle
// (a, b, inf) whose "circumcircle" is the open half-plane beyond the edge
// plus the open edge itself, so no finite super-triangle can perturb the
// hull.  Points are inserted along a Z-order curve and located by walking
// from the previous insertion, so each insertion touches O(1) triangles on
// average.  On co-circular points the in-circle test is strict, so the
// result is one of the valid Delaunay triangulations.
//
// Points of an image (coordinates below 2^14) take the in-circle test in 64-bit
// integers, which hold it exactly; an insertion allocates nothing (its lists are
// kept between insertions, and the cavity's fan is linked through the vertex at
// which each boundary edge starts and ends); the curve's keys are computed once.
// The 21754 points of a 752x480 keyframe, Grace host: 45.1 -> 8.0 ms.
#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

#include "gs.h"

namespace {

struct Tri {
    int v[3];   // counter-clockwise; -1 = the vertex at infinity (always v[2])
    int nb[3];  // neighbour across the edge opposite v[i]
    int mark;   // insertion stamp of the cavity search
    bool alive;
};

using i64 = long long;
using i128 = __int128;

// INT: the integer type that holds the in-circle determinant exactly -- below
// 3 |d|^2 |d|^2 for coordinate differences d: 64 bits up to 2^14, else 128.
template <class INT>
struct Del {
    const int32_t* xy;
    std::vector<Tri> t;
    // lists of one insertion, and by vertex (+ 1: the vertex at infinity first) the
    // new triangle whose boundary edge starts or ends there
    struct Edge { int a, b, outside; };
    std::vector<int> bad, stack, starts, ends;
    std::vector<Edge> edges;
    int stamp = 0;

    i64 X(int i) const { return xy[2 * i]; }
    i64 Y(int i) const { return xy[2 * i + 1]; }

    i64 orient(int a, int b, int c) const {
        return (X(b) - X(a)) * (Y(c) - Y(a)) - (Y(b) - Y(a)) * (X(c) - X(a));
    }

    // > 0: d strictly inside the circle through the CCW triangle a, b, c
    bool incircle(int a, int b, int c, int d) const {
        const i64 adx = X(a) - X(d), ady = Y(a) - Y(d);
        const i64 bdx = X(b) - X(d), bdy = Y(b) - Y(d);
        const i64 cdx = X(c) - X(d), cdy = Y(c) - Y(d);
        const INT al = (INT)adx * adx + (INT)ady * ady;
        const INT bl = (INT)bdx * bdx + (INT)bdy * bdy;
        const INT cl = (INT)cdx * cdx + (INT)cdy * cdy;
        const INT det = (INT)adx * ((INT)bdy * cl - (INT)cdy * bl) -
                        (INT)ady * ((INT)bdx * cl - (INT)cdx * bl) +
                        al * ((INT)bdx * cdy - (INT)cdx * bdy);
        return det > 0;
    }

    // p in the circumcircle of triangle k (the half-plane test for ghosts)
    bool in_circum(int k, int p) const {
        const Tri& T = t[k];
        if (T.v[2] >= 0) return incircle(T.v[0], T.v[1], T.v[2], p);
        const int a = T.v[0], b = T.v[1];
        const i64 o = orient(a, b, p);
        if (o != 0) return o > 0;
        // on the hull line: inside iff strictly between a and b
        const i64 d = (X(p) - X(a)) * (X(b) - X(a)) + (Y(p) - Y(a)) * (Y(b) - Y(a));
        const i64 l = (X(b) - X(a)) * (X(b) - X(a)) + (Y(b) - Y(a)) * (Y(b) - Y(a));
        return d > 0 && d < l;
    }

    // A triangle (real or ghost) whose circumcircle contains p, found by a
    // visibility walk from triangle `start`.
    int locate(int start, int p) const {
        int k = start;
        for (long long steps = 0; steps < (long long)4 * (long long)t.size() + 16; ++steps) {
            const Tri& T = t[k];
            if (T.v[2] < 0) return k;  // a ghost: p is beyond the hull edge (or on it)
            int next = -1;
            for (int i = 0; i < 3 && next < 0; ++i) {
                const int a = T.v[(i + 1) % 3], b = T.v[(i + 2) % 3];
                if (orient(a, b, p) < 0) next = T.nb[i];
            }
            if (next < 0) return k;  // p inside or on the boundary of T
            k = next;
        }
        return -1;  // cannot happen for a valid triangulation; reported as an error
    }

    int add(int a, int b, int c) {
        t.push_back(Tri{{a, b, c}, {-1, -1, -1}, 0, true});
        return (int)t.size() - 1;
    }

    // edge (a -> b) of triangle k: index of the opposite vertex
    static int edge_index(const Tri& T, int a, int b) {
        for (int i = 0; i < 3; ++i)
            if (T.v[(i + 1) % 3] == a && T.v[(i + 2) % 3] == b) return i;
        return -1;
    }

    // Inserts p; returns a new triangle containing p, or -1 on failure.
    int insert(int start, int p) {
        const int k0 = locate(start, p);
        if (k0 < 0 || !in_circum(k0, p)) return -1;
        ++stamp;
        bad.assign(1, k0);
        stack.assign(1, k0);
        t[k0].mark = stamp;
        while (!stack.empty()) {
            const int k = stack.back();
            stack.pop_back();
            for (int i = 0; i < 3; ++i) {
                const int q = t[k].nb[i];
                if (q < 0 || t[q].mark == stamp) continue;
                if (in_circum(q, p)) {
                    t[q].mark = stamp;
                    bad.push_back(q);
                    stack.push_back(q);
                }
            }
        }
        // the cavity's boundary edges, each turned into a triangle with p
        edges.clear();
        for (int k : bad) {
            Tri& T = t[k];
            for (int i = 0; i < 3; ++i) {
                const int q = T.nb[i];
                if (q >= 0 && t[q].mark == stamp) continue;
                edges.push_back({T.v[(i + 1) % 3], T.v[(i + 2) % 3], q});
            }
            T.alive = false;
        }
        int last = -1;
        const int first = (int)t.size();
        for (const Edge& e : edges) {
            // triangle (a, b, p), with the infinite vertex rotated last
            int k;
            if (e.a < 0) k = add(e.b, p, -1);
            else if (e.b < 0) k = add(p, e.a, -1);
            else k = add(e.a, e.b, p);
            Tri& T = t[k];
            // the outside neighbour across edge (a, b)
            T.nb[edge_index(T, e.a, e.b)] = e.outside;
            if (e.outside >= 0) {
                const int j = edge_index(t[e.outside], e.b, e.a);
                if (j >= 0) t[e.outside].nb[j] = k;
            }
            starts[e.a + 1] = k;
            ends[e.b + 1] = k;
            if (T.v[2] >= 0) last = k;
        }
        // link the fan: the boundary is one closed walk around p, so across
        // (b, p) lies the triangle whose edge starts at b, across (p, a) the one
        // whose edge ends at a
        for (size_t s = 0; s < edges.size(); ++s) {
            Tri& T = t[first + (int)s];
            const Edge& e = edges[s];
            T.nb[edge_index(T, e.b, p)] = starts[e.b + 1];
            T.nb[edge_index(T, p, e.a)] = ends[e.a + 1];
        }
        return last >= 0 ? last : (int)t.size() - 1;
    }
};

uint64_t morton(int32_t x, int32_t y) {
    uint64_t m = 0;
    for (int b = 0; b < 21; ++b)
        m |= ((uint64_t)((x >> b) & 1) << (2 * b)) | ((uint64_t)((y >> b) & 1) << (2 * b + 1));
    return m;
}

template <class INT>
gs_status triangulate(const int32_t* xy_host, int32_t n, int32_t* tri_host, int32_t tri_capacity,
                      int32_t* n_tri) {
    // along the curve, equal points (an error) next to each other
    std::vector<std::pair<uint64_t, int>> order(n);
    for (int i = 0; i < n; ++i) order[i] = {morton(xy_host[2 * i], xy_host[2 * i + 1]), i};
    std::sort(order.begin(), order.end());
    for (int i = 1; i < n; ++i)
        if (order[i].first == order[i - 1].first) return GS_ERR_INVALID;  // duplicate points
    Del<INT> d;
    d.xy = xy_host;
    d.t.reserve((size_t)6 * n + 16);
    d.starts.assign((size_t)n + 1, -1);
    d.ends.assign((size_t)n + 1, -1);
    // first triangle: the first point, the next one, and the first point off
    // their line (points before it are collinear and inserted afterwards)
    const int a = order[0].second, b = order[1].second;
    int c_pos = -1;
    for (int i = 2; i < n && c_pos < 0; ++i)
        if (d.orient(a, b, order[i].second) != 0) c_pos = i;
    if (c_pos < 0) return GS_OK;  // all collinear: no triangle
    int c = order[c_pos].second;
    int A = a, Bv = b, C = c;
    if (d.orient(A, Bv, C) < 0) std::swap(Bv, C);
    const int t0 = d.add(A, Bv, C);
    // ghosts on the three hull edges, each (u, v, inf) with the outside left of u -> v
    const int g0 = d.add(Bv, A, -1), g1 = d.add(C, Bv, -1), g2 = d.add(A, C, -1);
    // neighbours of t0: across edge opposite A = (Bv, C) -> ghost (C, Bv)
    d.t[t0].nb[0] = g1;
    d.t[t0].nb[1] = g2;
    d.t[t0].nb[2] = g0;
    auto link_ghost = [&](int g, int prev, int next) {
        // ghost (u, v, inf): nb[2] across (u, v) is t0; nb[0] across (v, inf),
        // nb[1] across (inf, u)
        d.t[g].nb[2] = t0;
        d.t[g].nb[0] = next;
        d.t[g].nb[1] = prev;
    };
    // hull (clockwise as seen from outside): g0 = (Bv, A), g2 = (A, C), g1 = (C, Bv)
    link_ghost(g0, g1, g2);
    link_ghost(g2, g0, g1);
    link_ghost(g1, g2, g0);
    int last = t0;
    for (int i = 2; i < n; ++i) {
        if (i == c_pos) continue;
        const int r = d.insert(last, order[i].second);
        if (r < 0) return GS_ERR_INVALID;
        last = r;
    }
    int cnt = 0;
    for (const Tri& T : d.t) {
        if (!T.alive || T.v[2] < 0) continue;
        if (cnt < tri_capacity) {
            tri_host[3 * cnt] = T.v[0];
            tri_host[3 * cnt + 1] = T.v[1];
            tri_host[3 * cnt + 2] = T.v[2];
        }
        ++cnt;
    }
    *n_tri = cnt;
    return cnt > tri_capacity ? GS_ERR_CAPACITY : GS_OK;
}

}  // namespace

extern "C" gs_status gs_delaunay(const int32_t* xy_host, int32_t n, int32_t* tri_host,
                                 int32_t tri_capacity, int32_t* n_tri) {
    if (!xy_host || !n_tri || n < 0 || tri_capacity < 0 || (tri_capacity > 0 && !tri_host))
        return GS_ERR_INVALID;
    *n_tri = 0;
    int32_t most = 0;
    for (size_t i = 0; i < 2 * (size_t)n; ++i) {
        if (xy_host[i] < 0 || xy_host[i] >= (1 << 20)) return GS_ERR_INVALID;
        most = std::max(most, xy_host[i]);
    }
    if (n < 3) return GS_OK;
    return most < (1 << 14) ? triangulate<i64>(xy_host, n, tri_host, tri_capacity, n_tri)
                            : triangulate<i128>(xy_host, n, tri_host, tri_capacity, n_tri);
}
