// CPU driver of the proper coadd's cut into chunks of tiles and groups of pairs (proper.cu).
// usage: host_cut in out   (in: i32 [n][7] T, max_tiles, tiles, pairs, ps, shared, P_R wanted;
//                           out: i64 [n][4] tiles, group, bytes used, bytes of the pool)
#include <cstdio>
#include <cstdlib>
#include "proper.cu"

// library helpers the translation unit references (host driver only)
int argus_check_shape(const argus_shape&, size_t) { return 0; }
void argus_count_launch(int) {}
int argus_launch_status() { return 0; }

int main(int argc, char** argv) {
    if (argc < 3) return 2;
    FILE *f = fopen(argv[1], "rb"), *g = fopen(argv[2], "wb");
    if (!f || !g) return 1;
    int c[7];
    while (fread(c, 4, 7, f) == 7) {
        const size_t pool = pool_bytes(c[0], c[1]);
        const CoaddCut k = coadd_cut(c[0], c[2], c[3], c[4], c[5], c[6], pool);
        const size_t npsf = c[5] ? 1 : k.tiles;            // as run_coadd lays the pool out
        const size_t used = npsf * (k.group * (k.rows + k.filt) + k.den + k.dtab) + (size_t)k.tiles * (k.group * k.z + k.out);
        const long long out[4] = {k.tiles, k.group, (long long)used, (long long)pool};
        if (fwrite(out, 8, 4, g) != 4) return 1;
    }
    fclose(f);
    fclose(g);
    return 0;
}
