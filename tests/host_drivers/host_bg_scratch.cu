// CPU driver of the background map's scratch layout (background.cu).
// usage: host_bg_scratch n...   (prints fill, meshf, missing and bytes for each count of boxes)
#include <cstdio>
#include <cstdlib>
#include "background.cu"

// library helpers the translation unit references (host driver only)
int argus_check_shape(const argus_shape&, size_t) { return 0; }
void argus_count_launch(int) {}
int argus_launch_status() { return 0; }
int argus_check_ptr16(const void*) { return 0; }

int main(int argc, char** argv) {
    for (int i = 1; i < argc; i++) {
        const BgScratch s = bg_scratch((size_t)atoll(argv[i]));
        printf("%zu %zu %zu %zu\n", s.fill, s.meshf, s.missing, s.bytes);
    }
    return 0;
}
