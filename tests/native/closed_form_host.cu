// The closed form of the cell integrals (field_common.cuh) run on the CPU:
// reads n, then per case FP64 vertices [9] and a point [3]; writes phi, F for
// both forms (geometry per evaluation and precomputed), for the precomputed form
// with the C library's functions, and the sum of the distances that multiply
// its logarithms and solid angle; and the helpers' sqrt, log ratio and arc
// tangent of three of the numbers.
#include "../../paper_2110_09214_gb300/csrc/obem_internal.cuh"
#include "../../paper_2110_09214_gb300/csrc/field_common.cuh"
#include <stdio.h>
#include <math.h>
#include <vector>

static void geo64(const double *v, double *g)
{
    const double e1[3] = {v[3] - v[0], v[4] - v[1], v[5] - v[2]}, e2[3] = {v[6] - v[0], v[7] - v[1], v[8] - v[2]};
    double n[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
    const double a2 = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    for (int k = 0; k < 3; ++k) g[k] = n[k] / a2;
    g[3] = a2;
    for (int e = 0; e < 3; ++e) {
        const int j = (e + 1) % 3;
        double d[3], *o = g + 4 + 6 * e;
        for (int k = 0; k < 3; ++k) d[k] = v[3 * j + k] - v[3 * e + k];
        const double len = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
        for (int k = 0; k < 3; ++k) o[k] = d[k] / len;
        o[3] = o[1] * g[2] - o[2] * g[1];
        o[4] = o[2] * g[0] - o[0] * g[2];
        o[5] = o[0] * g[1] - o[1] * g[0];
    }
}

// tri_closed_form_g with the C library's sqrt, log and atan2
static double plain(const double *v, const double *g, const double *r, double &phi, double *F)
{
    double a[3][3], R[3];
    for (int i = 0; i < 3; ++i) {
        for (int k = 0; k < 3; ++k) a[i][k] = v[3 * i + k] - r[k];
        R[i] = sqrt(a[i][0] * a[i][0] + a[i][1] * a[i][1] + a[i][2] * a[i][2]);
    }
    const double h = -(a[0][0] * g[0] + a[0][1] * g[1] + a[0][2] * g[2]);
    double scale = fabs(h);
    phi = F[0] = F[1] = F[2] = 0.0;
    for (int i = 0; i < 3; ++i) {
        const int j = (i + 1) % 3;
        const double *e = g + 4 + 6 * i;
        const double lm = a[i][0] * e[0] + a[i][1] * e[1] + a[i][2] * e[2];
        const double lp = a[j][0] * e[0] + a[j][1] * e[1] + a[j][2] * e[2];
        const double p0 = a[i][0] * e[3] + a[i][1] * e[4] + a[i][2] * e[5];
        double L;
        if (lm >= 0.0) L = log((R[j] + lp) / (R[i] + lm));
        else if (lp <= 0.0) L = log((R[i] - lm) / (R[j] - lp));
        else L = log((R[j] + lp) * (R[i] - lm) / (p0 * p0 + h * h));
        if (p0 != 0.0) phi += p0 * L;
        for (int k = 0; k < 3; ++k) F[k] += e[3 + k] * L;
        scale += fabs(p0);
    }
    auto dot = [&](int i, int j) { return a[i][0] * a[j][0] + a[i][1] * a[j][1] + a[i][2] * a[j][2]; };
    const double D = R[0] * R[1] * R[2] + dot(0, 1) * R[2] + dot(0, 2) * R[1] + dot(1, 2) * R[0];
    const double om = h == 0.0 ? 0.0 : 2.0 * atan2(g[3] * h, D);
    phi -= h * om;
    for (int k = 0; k < 3; ++k) F[k] += om * g[k];
    return scale;
}

int main(int argc, char **argv)
{
    if (argc < 3) return 2;
    FILE *f = fopen(argv[1], "rb"), *o = fopen(argv[2], "wb");
    int n = 0;
    if (!f || !o || fread(&n, 4, 1, f) != 1) return 2;
    std::vector<double> in(12 * (size_t)n);
    if (fread(in.data(), 8, in.size(), f) != in.size()) return 2;
    for (int i = 0; i < n; ++i) {
        const double *v = &in[12 * (size_t)i], *r = v + 9;
        double g[24], out[16];
        geo64(v, g);
        tri_closed_form(v, r[0], r[1], r[2], out[0], out[1], out[2], out[3]);
        tri_closed_form_g(v, g, r[0], r[1], r[2], out[4], out[5], out[6], out[7]);
        out[12] = plain(v, g, r, out[8], out + 9);
        out[13] = cf_sqrt(fabs(v[0]));
        out[14] = cf_log_ratio(fabs(v[1]), fabs(v[2]));
        out[15] = cf_atan2(v[3], v[4]);
        fwrite(out, 8, 16, o);
    }
    fclose(o);
    return 0;
}
