// Host side of the orbit tables (see orbit.h).
#include "orbit.h"

#include <algorithm>
#include <cmath>
#include <cstring>

#include "host_common.h"

namespace air {

namespace {

// A symmetry of the square about its centre as a signed permutation matrix.
struct Sym {
    int a, b, c, d;   // (x, y) -> (a x + b y, c x + d y)
};
Sym mul(const Sym &p, const Sym &q) {   // p after q
    return {p.a * q.a + p.b * q.c, p.a * q.b + p.b * q.d, p.c * q.a + p.d * q.c, p.c * q.b + p.d * q.d};
}
Sym inverse(const Sym &p) { return {p.a, p.c, p.b, p.d}; }   // orthogonal
int det(const Sym &p) { return p.a * p.d - p.b * p.c; }
// code -> matrix: exchange x and y first (ORB_T), then turn the axes (ORB_FX, ORB_FY)
Sym sym_of(int code) {
    const int sx = code & ORB_FX ? -1 : 1, sy = code & ORB_FY ? -1 : 1;
    return code & ORB_T ? Sym{0, sx, sy, 0} : Sym{sx, 0, 0, sy};
}
int code_of(const Sym &p) {
    const bool t = p.a == 0;
    const int sx = t ? p.b : p.a, sy = t ? p.c : p.d;
    return (t ? ORB_T : 0) | (sx < 0 ? ORB_FX : 0) | (sy < 0 ? ORB_FY : 0);
}

// An element of the scan's group: the symmetry, and what it does to view v:
// (sign v + shift) mod V, the bins reversed for sign -1.
struct Elem {
    Sym s;
    int sign, shift;
};

std::vector<Elem> scan_group(const air_geometry &g) {
    const int V = g.n_views;
    std::vector<Elem> G;
    if (std::fabs(g.arc - 2.0 * M_PI) > 1e-12 * 2.0 * M_PI) return G;
    const Sym turn{0, -1, 1, 0}, mirror{1, 0, 0, -1};
    const double m = -2.0 * g.beta0 * V / (2.0 * M_PI);      // mirrored view of view 0
    const bool mirrors = std::fabs(m) < 1e9 && std::fabs(m - std::nearbyint(m)) < 1e-9;
    const int m0 = mirrors ? (int)(((long long)std::nearbyint(m) % V + V) % V) : 0;
    Sym r{1, 0, 0, 1};
    for (int k = 0; k < 4; ++k) {
        if ((long long)k * V % 4 == 0) {
            const int shift = (int)((long long)k * V / 4);
            G.push_back({r, 1, shift});
            if (mirrors) G.push_back({mul(r, mirror), -1, (m0 + shift) % V});
        }
        r = mul(turn, r);
    }
    return G;
}

int map_view(const Elem &e, int v, int V) { return ((e.sign * v + e.shift) % V + V) % V; }

}  // namespace

void build_fbp_orbits(const air_geometry &g, FbpOrbits &T) {
    T = FbpOrbits();
    const std::vector<Elem> G = scan_group(g);
    if (G.size() != 4 && G.size() != 8) return;
    const int V = g.n_views;
    T.nf = (int)G.size();
    for (int f = 0; f < T.nf; ++f) T.code[f] = code_of(G[f].s);
    std::vector<char> seen(V, 0);
    for (int v = 0; v < V; ++v) {
        if (seen[v]) continue;
        T.base.push_back(v);
        for (int f = 0; f < 8; ++f) {
            const int w = f < T.nf ? map_view(G[f], v, V) : 0;
            T.view.push_back(f >= T.nf || seen[w] ? FBP_NONE : (G[f].sign < 0 ? ~w : w));
            if (f < T.nf) seen[w] = 1;
        }
    }
}

int orbit_frames(const air_geometry &g) {
    if (g.n < ORB_MIN_N) return 0;
    const size_t order = scan_group(g).size();
    return order == 4 || order == 8 ? (int)order : 0;
}

void build_orbits(const air_geometry &g, double dg, OrbitTables &T) {
    T = OrbitTables();
    const int nf = orbit_frames(g);
    if (!nf) return;
    const int n = g.n, V = g.n_views, nb = g.n_bins;
    const std::vector<Elem> G = scan_group(g);
    const double jm = 0.5 * (nb - 1), inv_dx = 1.0 / g.pixel_mm, half = 0.5 * n;
    // the fan stays well ahead of the source, so a line meets the image on
    // one side of it, and its rays are not much denser than the pixels
    if (jm * dg > 1.4) return;
    const double rmin = g.dso_mm * inv_dx - n / std::sqrt(2.0), rmax = g.dso_mm * inv_dx + n / std::sqrt(2.0);
    // a pixel's first candidate ray: the index's error in FP32 (source and
    // pixel coordinates up to rmax, the arctangent's series) and the third
    // order of the angle over the half diagonal of a warp's 8 x 16 pixels
    // (derivatives up to 2 / r^3)
    const double eps = 0.005 + (1.5e-6 * rmax / rmin + 206.0 / (rmin * rmin * rmin)) / dg;
    if (!(eps < 0.2)) return;

    // the classes' frames: the cosets of the group
    std::vector<int> frames[2];
    int class_of[8];
    std::fill(class_of, class_of + 8, -1);
    int nclass = 0;
    for (int c = 0; c < 8; ++c) {
        if (class_of[c] >= 0) continue;
        for (const Elem &e : G) class_of[code_of(mul(sym_of(c), e.s))] = nclass;
        for (int f = 0; f < 8; ++f)
            if (class_of[f] == nclass) frames[nclass].push_back(f);
        ++nclass;
    }

    struct View { int first, count; };             // rays of a base view
    std::vector<View> views;
    struct Seg { OrbSeg d; double sx, sy, cx, cy, ioff; int cls; };
    std::vector<Seg> segs;
    std::vector<RayFx> rays;
    std::vector<uint2> info;
    std::vector<char> seen(V, 0);
    for (int v = 0; v < V; ++v) {
        if (seen[v]) continue;
        int fixed = 0;
        for (const Elem &e : G) {
            const int w = map_view(e, v, V);
            seen[w] = 1;
            fixed += w == v;
        }
        const double beta = g.beta0 + g.arc * (double)v / (double)V;
        const double Sx = g.dso_mm * std::cos(beta), Sy = g.dso_mm * std::sin(beta);
        // a mirrored view takes itself to itself: half of its bins, and its
        // middle bin (odd counts), whose orbit has each ray twice, by itself
        std::vector<std::pair<int, int>> runs;
        if (fixed > 1) {
            if (nb / 2 > 0) runs.push_back({0, nb / 2});
            if (nb & 1) runs.push_back({nb / 2, nb / 2 + 1});
        } else {
            runs.push_back({0, nb});
        }
        const int first = (int)rays.size();
        for (const auto &run : runs) {
            auto frame_of = [&](int j) {
                const double th = beta + M_PI + ((double)j - jm) * dg;
                double a = std::cos(th), b = std::sin(th);
                const int t = std::fabs(b) > std::fabs(a) ? ORB_T : 0;
                if (t) std::swap(a, b);
                return t | (a < 0.0 ? ORB_FX : 0) | (b < 0.0 ? ORB_FY : 0);
            };
            for (int j0 = run.first; j0 < run.second;) {
                const int code = frame_of(j0);
                int j1 = j0 + 1;
                while (j1 < run.second && frame_of(j1) == code) ++j1;
                const Sym h = sym_of(code);
                const bool asc = det(h) > 0;
                const int cls = class_of[code];
                Seg S{};
                S.cls = cls;
                S.sx = (h.a * Sx + h.b * Sy) * inv_dx + half;
                S.sy = (h.c * Sx + h.d * Sy) * inv_dx + half;
                S.cx = -(h.a * std::cos(beta) + h.b * std::sin(beta));
                S.cy = -(h.c * std::cos(beta) + h.d * std::sin(beta));
                S.ioff = asc ? jm - j0 : (double)(j1 - 1) - jm;
                S.d.ray0 = (int)rays.size();
                S.d.cnt = j1 - j0;
                S.d.cls = cls;
                const bool middle = fixed > 1 && j0 == nb / 2;    // the run of one middle bin
                std::vector<int> taken;
                for (int f = 0; f < nf; ++f) {
                    // the member in frame f is g ray with frame[f] g = h
                    const Sym gs = mul(inverse(sym_of(frames[cls][f])), h);
                    const Elem *e = nullptr;
                    for (const Elem &q : G)
                        if (code_of(q.s) == code_of(gs)) e = &q;
                    if (!e) return;                               // not reached: frames are a coset of G
                    const int w = map_view(*e, v, V);
                    const bool up = (e->sign > 0) == asc;         // its bins ascend along the segment
                    const int jfirst = asc ? j0 : j1 - 1;         // base bin of the segment's ray 0
                    const int jf = e->sign > 0 ? jfirst : nb - 1 - jfirst;
                    S.d.zoff[f] = w * nb + jf;
                    if (!up) S.d.down |= 1 << f;
                    if (middle) {                                 // each ray of the orbit once
                        if (std::find(taken.begin(), taken.end(), S.d.zoff[f]) != taken.end()) S.d.zoff[f] = -1;
                        else taken.push_back(S.d.zoff[f]);
                    }
                }
                for (int i = 0; i < S.d.cnt; ++i) {
                    const int j = asc ? j0 + i : j1 - 1 - i;
                    const double th = beta + M_PI + ((double)j - jm) * dg;
                    const double ux = std::cos(th), uy = std::sin(th);
                    const double su = Sx * ux + Sy * uy;
                    const double px = (Sx - su * ux) * inv_dx, py = (Sy - su * uy) * inv_dx;
                    unsigned walk = 0;
                    const RayFx r = make_ray_fx(h.a * px + h.b * py + half, h.c * px + h.d * py + half,
                                                std::fabs(h.a * ux + h.b * uy), std::fabs(h.c * ux + h.d * uy), n, &walk);
                    // exchanged axes at a slope of one: keep the ray walking columns
                    if (!walk_cols(walk) || r.cs < 0.f) return;
                    // a ray along a grid line belongs to its + side, which a
                    // symmetry may take to the - side
                    const unsigned frac = (unsigned)(r.L0 + 2);
                    if (r.Mlo <= 1u && frac <= 4u) return;
                    const int k0 = walk_k0(walk), k1 = walk_k1(walk);
                    for (int k : {k0, k1 - 1}) {
                        if (k0 == k1) break;
                        const long long r0 = (r.L0 + (long long)k * ray_M(r)) >> 32;
                        if (k0 < 0 || k1 > n || r0 < -1 || r0 > n - 1) return;
                    }
                    rays.push_back(r);
                    info.push_back(make_uint2(walk, (unsigned)segs.size()));
                }
                segs.push_back(S);
                j0 = j1;
            }
        }
        views.push_back({first, (int)rays.size() - first});
    }
    if (rays.size() >= (1u << 26)) return;

    // segments in class order (rays stay where they are)
    std::vector<int> order(segs.size()), place(segs.size());
    for (size_t i = 0; i < segs.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return segs[a].cls < segs[b].cls; });
    for (size_t i = 0; i < order.size(); ++i) place[order[i]] = (int)i;
    for (uint2 &w : info) w.y = (unsigned)place[w.y];
    std::vector<Seg> sorted;
    for (int i : order) sorted.push_back(segs[i]);
    if (sorted.size() >= (1u << 17)) return;
    // the padded rays of the backprojector: a tile's candidates may run past
    // a segment's last ray, onto empty ones that add nothing
    std::vector<uint4> bray;
    for (Seg &S : sorted) {
        S.d.pad0 = (int)bray.size();
        for (int i = 0; i < S.d.cnt; ++i) {
            const RayFx &r = rays[S.d.ray0 + i];
            bray.push_back(make_uint4((unsigned)r.L0, (unsigned)((unsigned long long)r.L0 >> 32), r.Mlo, 0u));
        }
        bray.insert(bray.end(), ORB_CAND, make_uint4(0u, 0u, 0u, 0u));
    }

    // projector warps: up to 32 neighbouring rays each.  Groups of ORB_VIEWS
    // neighbouring base views at the same place of the fan, whose rays walk
    // neighbouring paths, stay together; the groups run from the longest walks
    // to the shortest, so that the last ones to finish are short
    struct Group { long long work; std::vector<unsigned> task; };
    std::vector<Group> groups;
    for (size_t v0 = 0; v0 < views.size(); v0 += ORB_VIEWS) {
        const size_t v1 = std::min(views.size(), v0 + ORB_VIEWS);
        int most = 0;
        for (size_t v = v0; v < v1; ++v) most = std::max(most, views[v].count);
        for (int c = 0; c < most; c += 32) {
            Group G1{0, {}};
            for (size_t v = v0; v < v1; ++v) {
                if (c >= views[v].count) continue;
                const int i0 = views[v].first + c, m = std::min(32, views[v].count - c);
                int ka = n, kb = 0;
                for (int i = i0; i < i0 + m; ++i)
                    if (walk_k0(info[i].x) < walk_k1(info[i].x)) {
                        ka = std::min(ka, walk_k0(info[i].x));
                        kb = std::max(kb, walk_k1(info[i].x));
                    }
                G1.work += std::max(0, kb - ka);
                G1.task.push_back((unsigned)i0 | (unsigned)(m - 1) << 26);
            }
            groups.push_back(G1);
        }
    }
    std::stable_sort(groups.begin(), groups.end(), [](const Group &a, const Group &b) { return a.work > b.work; });
    std::vector<unsigned> task;
    for (const Group &G1 : groups) task.insert(task.end(), G1.task.begin(), G1.task.end());

    // backprojector: per class and 32 x 32 canonical pixel tile the segments
    // with rays that meet it: the rays whose angle lies between the extreme
    // angles of the tile's corners, widened by 0.02 ray, and the most rays
    // that can meet two pixels of a column (their width across a ray over the
    // tile's distance from the source)
    const int tpr = (n + BWD_T - 1) / BWD_T, nt = tpr * tpr;
    std::vector<int> tile0(2 * (size_t)(nt + 1), 0);
    std::vector<std::vector<uint2>> lists(2 * (size_t)nt);
    std::vector<double> angle((size_t)(tpr + 1) * (tpr + 1)), width(angle.size());   // at the tiles' corners
    for (size_t si = 0; si < sorted.size(); ++si) {
        const Seg &S = sorted[si];
        for (int iy = 0; iy <= tpr; ++iy)
            for (int ix = 0; ix <= tpr; ++ix) {
                const double ex = std::min(n, ix * BWD_T) - S.sx, ey = std::min(n, iy * BWD_T) - S.sy;
                const size_t i = (size_t)iy * (tpr + 1) + ix;
                angle[i] = std::atan2(S.cx * ey - S.cy * ex, S.cx * ex + S.cy * ey);
                width[i] = (2.0 * std::fabs(ex) + std::fabs(ey)) / std::sqrt(ex * ex + ey * ey);
            }
        for (int ty = 0; ty < tpr; ++ty)
            for (int tx = 0; tx < tpr; ++tx) {
                const double x0 = tx * BWD_T, x1 = std::min(n, (tx + 1) * BWD_T);
                const double y0 = ty * BWD_T, y1 = std::min(n, (ty + 1) * BWD_T);
                double gmin = 1e30, gmax = -1e30, wide = 0.0;
                for (int cy = ty; cy <= ty + 1; ++cy)
                    for (int cx = tx; cx <= tx + 1; ++cx) {
                        const size_t i = (size_t)cy * (tpr + 1) + cx;
                        gmin = std::min(gmin, angle[i]);
                        gmax = std::max(gmax, angle[i]);
                        wide = std::max(wide, width[i]);
                    }
                const double f0 = std::ceil(gmin / dg + S.ioff - 0.02), f1 = std::floor(gmax / dg + S.ioff + 0.02);
                const int a = (int)std::max(0.0, std::min(f0, (double)S.d.cnt));
                const int b = (int)std::max(-1.0, std::min(f1, (double)S.d.cnt - 1.0)) + 1;
                if (b <= a) continue;
                const double nx = std::min(std::max(S.sx, x0), x1) - S.sx, ny = std::min(std::max(S.sy, y0), y1) - S.sy;
                const double most = std::min(wide + 0.1, std::sqrt(5.0)) / std::hypot(nx, ny) / dg;
                const double cand = std::floor(most + 2.0 * eps) + 1.0;
                if (b - a > ORB_RAYS || cand > ORB_CAND) return;
                lists[(size_t)S.cls * nt + ty * tpr + tx].push_back(
                    make_uint2((unsigned)si | (unsigned)(b - a) << 17 | (unsigned)cand << 24, (unsigned)(S.d.pad0 + a)));
            }
    }
    std::vector<uint2> ent;
    for (int c = 0; c < 2; ++c)
        for (int t = 0; t <= nt; ++t) {
            tile0[(size_t)c * (nt + 1) + t] = (int)ent.size();
            if (t < nt) ent.insert(ent.end(), lists[(size_t)c * nt + t].begin(), lists[(size_t)c * nt + t].end());
        }

    std::vector<uint2> zmap((size_t)V * nb);
    for (const Seg &S : sorted)
        for (int f = 0; f < nf; ++f)
            for (int i = 0; i < S.d.cnt && S.d.zoff[f] >= 0; ++i) {
                unsigned c;
                std::memcpy(&c, &rays[S.d.ray0 + i].cs, 4);
                zmap[S.d.zoff[f] + ((S.d.down >> f) & 1 ? -i : i)] =
                    make_uint2((unsigned)((f / 4) * bray.size() + S.d.pad0 + i) * 4u + (unsigned)(f & 3), c);
            }

    T.eps = (float)eps;
    for (size_t i = 0; i < sorted.size(); ++i) {
        OrbSeg d = sorted[i].d;
        d.sx = (float)sorted[i].sx;
        d.sy = (float)sorted[i].sy;
        d.cx = (float)sorted[i].cx;
        d.cy = (float)sorted[i].cy;
        d.ioff = (float)(sorted[i].ioff - eps);
        T.seg.push_back(d);
        T.nseg[d.cls] += 1;
    }
    for (int p = 0; p < 8; ++p) T.frame[p] = nf == 8 ? frames[0][p] : frames[p / 4][p % 4];
    T.ray = std::move(rays);
    T.info = std::move(info);
    T.task = std::move(task);
    T.tile0 = std::move(tile0);
    T.ent = std::move(ent);
    T.bray = std::move(bray);
    T.zmap = std::move(zmap);
    T.nf = nf;
}

}  // namespace air
