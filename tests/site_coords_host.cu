// The site coordinates of csrc/dlz_internal.cuh and wilson_eo_site.cuh by an operator's divisors, as
// device code computes them, exported for tests/test_site_coords_host.py
#include "wilson_eo_site.cuh"

using namespace dlz;

static Geom geom(const int *L) {
    Geom g{{L[0], L[1], L[2], L[3]}, L[0] * L[1] * L[2] * L[3], -1};
    g.set_divisors();
    return g;
}

// first site with other coordinates than s = ((t Lz + z) Ly + y) Lx + x says, or -1
extern "C" int coords_first_wrong(const int *L, int first, int count) {
    const Geom g = geom(L);
    for (int s = first; s < first + count; ++s) {
        int c[4];
        site_coords(g, s, c);
        for (int i = 0, r = s; i < 4; r /= L[i], ++i)
            if (c[i] != (i < 3 ? r % L[i] : r)) return s;
    }
    return -1;
}

// the same for the checkerboard: the sites of parity `par` in order, L[0] even
extern "C" int eo_first_wrong(const int *L, int par) {
    const Geom g = geom(L);
    int cb = 0;
    for (int s = 0; s < g.V; ++s) {
        int w[4];
        for (int i = 0, r = s; i < 4; r /= L[i], ++i) w[i] = i < 3 ? r % L[i] : r;
        if (((w[0] + w[1] + w[2] + w[3]) & 1) != par) continue;
        int c[4];
        if (eo_site(cb, par, g, c) != s) return s;
        for (int i = 0; i < 4; ++i)
            if (c[i] != w[i]) return s;
        ++cb;
    }
    return -1;
}
