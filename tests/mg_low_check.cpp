// Test harness (host only): the V-cycle that the solver applies -- built on the
// second-order operator of the cell's stencil directions -- as preconditioner of CG on
// the sixth-order Poisson problem of one proto-subdomain, against the V-cycle built
// on that operator itself and against plain CG.  Prints one JSON line.
//   usage: mg_low_check scale s1 s2 n R_PE R_ME fd_n
#define main mg_check_main
#include "mg_check.cpp"
#undef main

int main(int argc, char **argv)
{
    if (argc < 8) return 2;
    const double scale = std::atof(argv[1]), s1 = std::atof(argv[2]), s2 = std::atof(argv[3]);
    const int ng = std::atoi(argv[4]), fd = std::atoi(argv[7]);
    const double rpe = std::atof(argv[5]), rme = std::atof(argv[6]);
    const double lat[3][3] = {{scale, 0, 0}, {s1 * scale, scale, 0}, {s2 * scale, -s2 * 1.6 * scale, scale}};
    const int n[3] = {ng, ng, ng};
    Metric m;
    Stencil st;
    OffsetSet o;
    SetLayout L;
    if (make_metric(lat, n, m) || make_stencil(m, fd, 15, nullptr, 0, st) || make_offsets(m, rpe, rme, o) ||
        make_layout(o, st, fd, L))
        return 3;
    std::vector<MgLevel> lh, ll;
    MgTables th, tl;
    const double w = 0.8, sc = mg_omega_scale(fd);
    if (make_mg_levels(L, st, fd, 200, lh) || make_mg_levels(L, st, 1, 200, ll) ||
        make_mg_tables(L, st, fd, 200, w, 0.005, th) || make_mg_tables(L, st, 1, 200, w * sc, 0.005, tl))
        return 4;
    const MgLevel &A = lh[0];
    Vec b(A.n);
    unsigned seed = 12345;
    for (double &v : b) {
        seed = seed * 1664525u + 1013904223u;
        v = (seed >> 8) / 16777216.0 - 0.5;
    }
    auto cycle = [&](const MgTables &T, const MgLevel &f, double om) {
        double diag = 0.0;
        for (int k = f.row[0]; k < f.row[1]; ++k)
            if (f.col[k] == 0) diag = f.val[k];
        return MgT{&T, &f, (float)(om / diag)};
    };
    const MgT Mh = cycle(th, lh[0], w), Ml = cycle(tl, ll[0], w * sc);
    Vec x0, xh, xl;
    // (a set that is too small or whose coarse stencils reach too far has no hierarchy: -1)
    const int n0 = pcg<MgT>(A, b, nullptr, 1e-9, x0), nh = th.nlev ? pcg(A, b, &Mh, 1e-9, xh) : -1,
              nl = tl.nlev ? pcg(A, b, &Ml, 1e-9, xl) : -1;
    if (!tl.nlev) xl = x0;
    double d2 = 0.0, r2 = 0.0;
    for (int i = 0; i < A.n; ++i) {
        d2 += (xl[i] - x0[i]) * (xl[i] - x0[i]);
        r2 += x0[i] * x0[i];
    }
    std::printf("{\"definite\": %d, \"scale\": %.6f, \"plain\": %d, \"high\": %d, \"low\": %d, \"rel_diff\": %.3e, "
                "\"K1_high\": %d, \"K1_low\": %d}\n",
                (int)mg_definite(st), sc, n0, nh, nl, std::sqrt(d2 / r2), th.K[1], tl.K[1]);
    return 0;
}
