// The closed form of the cell integrals in pairs of floats (closed_form_df.cuh)
// run on the CPU beside the FP64 form: reads n, then per case FP64 vertices [9]
// and a binary32 point [3]; writes whether the pairs decided the case, phi and F
// of both forms.
#include "../../paper_2110_09214_gb300/csrc/obem_internal.cuh"
#include "../../paper_2110_09214_gb300/csrc/field_common.cuh"
#include <stdio.h>
#include <vector>

static void cross(const double *a, const double *b, double *c)
{
    for (int k = 0; k < 3; ++k) c[k] = a[(k + 1) % 3] * b[(k + 2) % 3] - a[(k + 2) % 3] * b[(k + 1) % 3];
}
static double unit(double *a)
{
    const double l = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
    for (int k = 0; k < 3; ++k) a[k] /= l;
    return l;
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
        double g[OBEM_GEO64] = {0}, e[3][3], out[9];
        for (int a = 0; a < 3; ++a)
            for (int k = 0; k < 3; ++k) e[a][k] = v[3 * ((a + 1) % 3) + k] - v[3 * a + k];
        const double m[3] = {-e[2][0], -e[2][1], -e[2][2]};
        cross(e[0], m, g);
        g[3] = unit(g);
        for (int a = 0; a < 3; ++a) {
            unit(e[a]);
            for (int k = 0; k < 3; ++k) g[4 + 6 * a + k] = e[a][k];
            cross(e[a], g, g + 7 + 6 * a);
        }
        float2 g2[OBEM_GEO2];
        for (int k = 0; k < OBEM_GEO2; ++k) {
            const double x = k < 9 ? v[k] : g[k - 9];
            g2[k] = make_float2((float)x, (float)(x - (double)(float)x));
        }
        Dbf q[4];
        out[0] = tri_closed_df(g2, Dbf{(float)r[0], 0.f}, Dbf{(float)r[1], 0.f}, Dbf{(float)r[2], 0.f}, true, q[0], q[1], q[2],
                               q[3]);
        for (int k = 0; k < 4; ++k) out[1 + k] = (double)q[k].h + (double)q[k].l;
        tri_closed_form_g(v, g, r[0], r[1], r[2], out[5], out[6], out[7], out[8]);
        fwrite(out, 8, 9, o);
    }
    fclose(o);
    return 0;
}
