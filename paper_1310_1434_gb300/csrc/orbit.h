// Orbit tables: the rays of a scan grouped by the symmetries of the pixel grid.
//
// The eight symmetries of the square (quarter turns and reflections) map the
// pixel grid onto itself, and a full rotation of equally spaced views onto
// itself as well: a quarter turn takes view v to v + V/4 (V a multiple of 4),
// a reflection takes it to a mirrored view with its bins reversed (beta0 a
// multiple of half the view pitch), a half turn to v + V/2.  The rays that
// such a group G takes into one another (an orbit, |G| of them) have the same
// lengths in the pixels that the same symmetries take into one another, so
// the integer arithmetic of one ray serves |G| rays.
//
// Every ray has one symmetry h of the square that makes it walk columns
// towards +x with a slope in [0, 1] (its canonical form); the rays of an orbit
// share that form and differ in h, their FRAME: the canonical ray meets the
// canonical pixel (k, r) where the physical ray meets the pixel h^-1 (k, r).
// The frames of an orbit are a coset of G.  With |G| = 8 there is one class of
// orbits with all eight frames, with |G| = 4 two classes of four.  Frames
// come in two PLANES of four: plane p of class 0 (|G| = 8), or of class p.
#pragma once

#include <vector>

#include "air_internal.cuh"

namespace air {

struct OrbitTables {
    int nf = 0;                       // frames per orbit, 8 or 4 (0: the scan does not qualify)
    int frame[8] = {};                // symmetry codes, plane-major (ORB_T | ORB_FX | ORB_FY)
    float eps = 0.f;                  // slack of a pixel's first candidate ray, in rays
    int nseg[2] = {0, 0};             // segments per class
    std::vector<OrbSeg> seg;          // class 0's, then class 1's
    std::vector<RayFx> ray;           // canonical rays, segment by segment, by ascending angle
    std::vector<uint2> info;          // per ray: {walk word, segment}
    std::vector<unsigned> task;       // projector warps: first ray | (rays - 1) << 26
    std::vector<int> tile0;           // [2 classes][pixel tiles + 1] offsets into ent
    std::vector<uint2> ent;           // backprojector: per class and tile the segments that meet it
    std::vector<uint4> bray;          // padded rays: each segment's, then ORB_CAND empty ones
    std::vector<uint2> zmap;          // per physical ray: place among the packed samples (floats), c
};

// The views of a full scan grouped by its symmetries, for the analytic
// reconstruction: what a pixel p takes from base view v, the pixel g p takes
// from view g v.  Slot f is symmetry code[f]; a mirrored view's bins are
// reversed; a base view that a mirror takes to itself has each view twice,
// of which one slot is left empty.
struct FbpOrbits {
    int nf = 0;                       // symmetries, 8 or 4 (0: fewer)
    int code[8] = {};
    std::vector<int> base;            // base views
    std::vector<int> view;            // [base][8]: view, ~view (reversed) or FBP_NONE
};
void build_fbp_orbits(const air_geometry &g, FbpOrbits &T);

// Frames per orbit of a scan with enough symmetries (8 or 4, else 0).
int orbit_frames(const air_geometry &g);

// Fills T, or leaves T.nf = 0 where the scan has fewer than four symmetries or
// its rays do not suit the orbit kernels.
void build_orbits(const air_geometry &g, double dg, OrbitTables &T);

}  // namespace air
