// CPU driver of the HEALPix patch path (healpix.cu): per half patch the nodes, the columns'
// cubics, their differences and the fixed-point positions, pixel by pixel beside the exact
// path's, and the fixed-point interpolation of four values.
// usage: host_hp_patch pos nside_seg k wcs segs out   (wcs: f64 [6], segs: i64 [n]; out: f64 [halves][32][64][4]
//                                                       positions from the patch and exact, halves in the belt only)
//        host_hp_patch lerp in out                     (in: f32 [n][4], then f64 [n][2] fractions; out: f32 [n])
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "healpix.cu"

// library helpers the translation unit references (host driver only)
int argus_check_shape(const argus_shape&, size_t) { return 0; }
void argus_count_launch(int) {}
int argus_launch_status() { return 0; }

static std::vector<char> slurp(const char* path) {
    FILE* f = fopen(path, "rb");
    if (!f) exit(1);
    std::vector<char> b;
    char q[65536];
    for (size_t n; (n = fread(q, 1, sizeof q, f)) > 0;) b.insert(b.end(), q, q + n);
    fclose(f);
    return b;
}

int main(int argc, char** argv) {
    if (argc < 4) return 2;
    FILE* g = fopen(argv[argc - 1], "wb");
    if (!g) return 1;
    if (!strcmp(argv[1], "lerp")) {
        const std::vector<char> b = slurp(argv[2]);
        const size_t n = b.size() / 32;
        const float* q = reinterpret_cast<const float*>(b.data());
        const double* t = reinterpret_cast<const double*>(b.data() + 16 * n);
        for (size_t i = 0; i < n; i++) {
            const float v = hp_fixed_bilinear(q[4 * i], q[4 * i + 1], q[4 * i + 2], q[4 * i + 3],
                                              (long long)(t[2 * i] * 0x1p44), (long long)(t[2 * i + 1] * 0x1p44));
            fwrite(&v, 4, 1, g);
        }
        fclose(g);
        return 0;
    }
    static constexpr HpWeights W = hp_make_weights();
    HpArgs a;
    memset(&a, 0, sizeof a);
    a.nside_seg = atoi(argv[2]);
    a.k = atoi(argv[3]);
    const std::vector<char> wb = slurp(argv[4]), sb = slurp(argv[5]);
    argus_wcs wcs;
    memcpy(&wcs, wb.data(), sizeof wcs);
    hp_fill_wcs(a, wcs);
    const int m = 1 << a.k;
    for (size_t s = 0; s < sb.size() / 8; s++) {
        const HpSeg sg = hp_seg(a, reinterpret_cast<const long long*>(sb.data())[s]);
        for (int r0 = 0; r0 < m; r0 += HP_HALF)
            for (int c0 = 0; c0 < m; c0 += HP_PATCH) {
                if (!hp_in_belt(sg, c0, r0, HP_PATCH, HP_HALF)) continue;
                double nd[4][4][2];
                for (int j = 0; j < 4; j++)
                    for (int i = 0; i < 4; i++) {
                        const int c = c0 + hp_node(i), r = r0 + hp_node_row(j);
                        if (!hp_on_ring(a, sg, c, r, hp_ring(sg.nside, sg.jr - c - r), nd[j][i][0], nd[j][i][1])) return 1;
                    }
                std::vector<double> out((size_t)HP_HALF * HP_PATCH * 4);
                for (int col = 0; col < HP_PATCH; col++)
                    for (int xy = 0; xy < 2; xy++) {
                        double v[4];
                        for (int j = 0; j < 4; j++) v[j] = hp_column(W.w[col], nd[j][0][xy], nd[j][1][xy], nd[j][2][xy], nd[j][3][xy]);
                        long long f[4], d[4];
                        hp_differences(v, f);
                        for (int r = 0; r < HP_HALF; r++) {
                            if (r % (HP_HALF / 4) == 0) hp_advance(f, r, d);
                            out[((size_t)r * HP_PATCH + col) * 4 + xy] = (double)d[0] * 0x1p-44;
                            hp_step(d);
                        }
                    }
                for (int r = 0; r < HP_HALF; r++)
                    for (int c = 0; c < HP_PATCH; c++) {
                        double* o = &out[((size_t)r * HP_PATCH + c) * 4];
                        if (!hp_on_ring(a, sg, c0 + c, r0 + r, hp_ring(sg.nside, sg.jr - c0 - c - r0 - r), o[2], o[3])) return 1;
                    }
                fwrite(out.data(), 8, out.size(), g);
            }
    }
    fclose(g);
    return 0;
}
