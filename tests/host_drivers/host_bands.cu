// CPU driver of the subtraction's choice of bands (subtract_tc.cu).
// usage: host_bands in out   (in: i32 [n][4] w, h, r, SMs; out: i32 [n][2] rows of a difference and a variance band)
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "subtract_tc.cu"

// library helpers the translation unit references (host driver only)
void argus_count_launch(int) {}
int argus_launch_status() { return 0; }
int argus_cuda_fail(cudaError_t) { return ARGUS_ERR_CUDA; }
int argus_tmap_2d(CUtensorMap*, CUtensorMapDataType, int, const void*, long, long, long, int, int) { return 0; }

int main(int argc, char** argv) {
    if (argc < 3) return 2;
    FILE *f = fopen(argv[1], "rb"), *g = fopen(argv[2], "wb");
    if (!f || !g) return 1;
    int c[4];
    while (fread(c, 4, 4, f) == 4) {
        const int out[2] = {band_rows<false>(c[0], c[1], c[2], c[3]), band_rows<true>(c[0], c[1], c[2], 2 * c[3])};
        if (fwrite(out, 4, 2, g) != 2) return 1;
    }
    fclose(f);
    fclose(g);
    return 0;
}
