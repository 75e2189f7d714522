// CPU driver of the clipped coadd's shift arithmetic (coadd.cu): split_shift per value and,
// for every pair of values, whether the windows' union fits the shared table.
// usage: host_coadd_shift size in out   (in: f32 [n]; out: i32 [n], f32 [n] fractions, f32 [2][n] weights, u8 [n][n])
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "coadd.cu"

// library helpers the translation unit references (host driver only)
int argus_check_shape(const argus_shape&, size_t) { return 0; }
int argus_check_ptr16(const void*) { return 0; }
void argus_count_launch(int) {}
int argus_launch_status() { return 0; }

int main(int argc, char** argv) {
    if (argc < 4) return 2;
    const int size = atoi(argv[1]);
    FILE* f = fopen(argv[2], "rb");
    if (!f) return 1;
    std::vector<float> v, frac, w0, w1;
    std::vector<int> whole;
    std::vector<unsigned char> fits;
    float x;
    while (fread(&x, 4, 1, f) == 1) v.push_back(x);
    fclose(f);
    for (float s : v) {
        const ShiftPart p = split_shift(s, size);
        whole.push_back(p.whole);
        frac.push_back(p.frac);
        w0.push_back(p.w0);
        w1.push_back(p.w1);
    }
    for (int a : whole)
        for (int b : whole) fits.push_back(union_fits(a > b ? a - b : b - a, 0) && union_fits(0, a > b ? a - b : b - a));
    FILE* g = fopen(argv[3], "wb");
    if (!g) return 1;
    fwrite(whole.data(), 4, whole.size(), g);
    fwrite(frac.data(), 4, frac.size(), g);
    fwrite(w0.data(), 4, w0.size(), g);
    fwrite(w1.data(), 4, w1.size(), g);
    fwrite(fits.data(), 1, fits.size(), g);
    fclose(g);
    return 0;
}
