// Host check of the orbit tables against the general ray table: no GPU needed.
// Usage: orbit_tables n pixel_mm views bins dso_mm beta0.  Prints the frames
// per orbit (0: the scan does not qualify) and exits with the number of faults.
//   - the projector's warps cover every canonical ray once, and the orbits
//     every physical ray once;
//   - each physical ray gets the same lengths (to 1e-4 px, the sensitivity of
//     nearly axis-parallel rays to the tables' 2^-32 px) in the same pixels as
//     from its own entry of the general table, the same in sum;
//   - the backprojector's lists, first candidates and candidate counts reach
//     every (ray, pixel) pair of the projector once, with the same overlap.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <unordered_map>
#include <vector>

#include "host_common.h"
#include "orbit.h"

using namespace air;

static void pixel(int code, int n, int k, int r, int &ix, int &iy) {
    const int a = code & ORB_FX ? n - 1 - k : k, b = code & ORB_FY ? n - 1 - r : r;
    ix = code & ORB_T ? b : a;
    iy = code & ORB_T ? a : b;
}

int main(int argc, char **argv) {
    if (argc < 7) return 255;
    air_geometry g{};
    g.n = std::atoi(argv[1]);
    g.pixel_mm = std::atof(argv[2]);
    g.n_views = std::atoi(argv[3]);
    g.n_bins = std::atoi(argv[4]);
    g.dso_mm = std::atof(argv[5]);
    g.beta0 = std::atof(argv[6]);
    g.arc = 2.0 * M_PI;
    const double dg = fan_pitch(g);
    const int n = g.n, V = g.n_views, nb = g.n_bins;
    OrbitTables T;
    build_orbits(g, dg, T);
    std::printf("%d\n", T.nf);
    if (!T.nf) return 0;
    int bad = 0;
    std::vector<int> warps(T.ray.size(), 0), rays((size_t)V * nb, 0);
    for (unsigned w : T.task)
        for (unsigned i = 0; i <= w >> 26; ++i) warps.at((w & 0x3ffffffu) + i) += 1;
    for (int c : warps) bad += c != 1;

    std::unordered_map<unsigned long long, unsigned> pairs;   // (ray, pixel) -> overlap
    for (size_t i = 0; i < T.ray.size(); ++i) {
        const RayFx &r = T.ray[i];
        const OrbSeg &s = T.seg[T.info[i].y];
        const int j = (int)i - s.ray0;
        for (int f = 0; f < T.nf; ++f) {
            if (s.zoff[f] < 0) continue;
            const int z = s.zoff[f] + ((s.down >> f) & 1 ? -j : j), v = z / nb, b = z % nb;
            rays.at(z) += 1;
            // the filter's place for this ray's sample is the backprojector's
            unsigned c;
            memcpy(&c, &r.cs, 4);
            bad += T.zmap.at(z).x != ((f / 4) * T.bray.size() + s.pad0 + j) * 4 + (f & 3) || T.zmap[z].y != c;
            const int code = T.frame[T.nf == 8 ? f : 4 * s.cls + f];
            std::map<int, double> diff;
            double sum = 0.0;
            for (int k = walk_k0(T.info[i].x); k < walk_k1(T.info[i].x); ++k) {
                const unsigned long long p = (unsigned long long)r.L0 + (unsigned long long)k * r.Mlo;
                const unsigned ov[2] = {std::min(r.Mlo, ~(unsigned)p), r.Mlo - std::min(r.Mlo, ~(unsigned)p)};
                for (int q = 0; q < 2; ++q) {
                    const int row = (int)(p >> 32) + q;
                    if (!ov[q] || row < 0 || row >= n) continue;
                    int ix, iy;
                    pixel(code, n, k, row, ix, iy);
                    pairs[(unsigned long long)z * n * n + (unsigned)(iy * n + ix)] = ov[q];
                    diff[iy * n + ix] += ov[q] * (double)r.cs;
                    sum += ov[q] * (double)r.cs;
                }
            }
            const double beta = g.beta0 + g.arc * v / V, th = beta + M_PI + (b - 0.5 * (nb - 1)) * dg;
            const double ux = std::cos(th), uy = std::sin(th), Sx = g.dso_mm * std::cos(beta), Sy = g.dso_mm * std::sin(beta);
            const double su = Sx * ux + Sy * uy;
            unsigned walk;
            const RayFx q = make_ray_fx((Sx - su * ux) / g.pixel_mm + 0.5 * n, (Sy - su * uy) / g.pixel_mm + 0.5 * n, ux, uy,
                                        n, &walk);
            for (int k = walk_k0(walk); k < walk_k1(walk); ++k) {
                const unsigned long long p = (unsigned long long)(q.L0 + k * ray_M(q));
                const unsigned Ma = ray_Ma(q), ov0 = std::min(Ma - 1u, ~(unsigned)p) + 1u;
                for (int h = 0; h < 2; ++h) {
                    const int row = (int)(p >> 32) + h;
                    const unsigned ov = h ? Ma - ov0 : ov0;
                    if (!ov || row < 0 || row >= n) continue;
                    diff[walk_cols(walk) ? row * n + k : k * n + row] -= ov * (double)std::fabs(q.cs);
                    sum -= ov * (double)std::fabs(q.cs);
                }
            }
            for (const auto &kv : diff) bad += std::fabs(kv.second) > 1e-4;
            bad += std::fabs(sum) > 1e-4;
        }
    }
    for (int c : rays) bad += c != 1;

    const int tpr = (n + BWD_T - 1) / BWD_T, nt = tpr * tpr;
    std::unordered_map<unsigned long long, int> got;
    for (int c = 0; c < 2; ++c)
        for (int t = 0; t < nt; ++t)
            for (int e = T.tile0[c * (nt + 1) + t]; e < T.tile0[c * (nt + 1) + t + 1]; ++e) {
                const uint2 w = T.ent[e];
                const OrbSeg &s = T.seg[w.x & 0x1ffffu];
                const int cand = (int)(w.x >> 24), cnt = (int)(w.x >> 17) & 0x7f, first = (int)w.y - s.pad0;
                bad += s.cls != c || cnt > ORB_RAYS || cand > ORB_CAND || w.y + cnt + ORB_CAND > T.bray.size();
                for (int k = (t % tpr) * BWD_T; k < std::min(n, (t % tpr + 1) * BWD_T); ++k)
                    for (int r = (t / tpr) * BWD_T; r < std::min(n, (t / tpr + 1) * BWD_T); r += 2) {
                        // first ray at or after the angle of the corner (k + 1, r), early by up to eps
                        const double X = k + 1 - (double)s.sx, Y = r - (double)s.sy;
                        const double idx = std::atan2(s.cx * Y - s.cy * X, s.cx * X + s.cy * Y) / dg + s.ioff - first;
                        for (const double early : {0.0, (double)T.eps}) {
                            const int i0 = std::min(std::max((int)std::ceil(idx + T.eps - early - 1e-3 * T.eps), 0), cnt);
                            for (int q = 0; q < cand; ++q) {
                                const uint4 ray = T.bray[w.y + i0 + q];
                                const unsigned long long p = (((unsigned long long)ray.y << 32) | ray.x) + (unsigned long long)k * ray.z;
                                const unsigned ov0 = std::min(ray.z, ~(unsigned)p), ov1 = ray.z - ov0;
                                const int d = (int)(p >> 32) - r, i = first + i0 + q;
                                for (int h = 0; h < 2; ++h) {
                                    const unsigned ov = d == h ? ov0 : (d == h - 1 ? ov1 : 0u);
                                    if (!ov || r + h >= n) continue;
                                    for (int f = 0; f < T.nf && i < s.cnt; ++f) {
                                        if (s.zoff[f] < 0) continue;
                                        int ix, iy;
                                        pixel(T.frame[T.nf == 8 ? f : 4 * c + f], n, k, r + h, ix, iy);
                                        const unsigned long long key =
                                            (unsigned long long)(s.zoff[f] + ((s.down >> f) & 1 ? -i : i)) * n * n +
                                            (unsigned)(iy * n + ix);
                                        const auto it = pairs.find(key);
                                        bad += it == pairs.end() || it->second != ov;
                                        got[key] += early == 0.0 ? 1 : 1 << 16;
                                    }
                                    bad += i >= s.cnt;
                                }
                            }
                        }
                    }
            }
    bad += got.size() != pairs.size();
    for (const auto &kv : got) bad += kv.second != 1 + (1 << 16);
    return bad > 200 ? 200 : bad;
}
