// CPU driver of the box medians' selection (background.cu): the bracket's passes over a
// box's keys, counted serially, and the three ways a selection ends.
// usage: host_box_median n in out   (in: f32 [boxes][n], NaN where invalid; out: f64 [boxes] medians, i32 [boxes] passes)
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include <vector>
#include "background.cu"

// library helpers the translation unit references (host driver only)
int argus_check_shape(const argus_shape&, size_t) { return 0; }
void argus_count_launch(int) {}
int argus_launch_status() { return 0; }
int argus_check_ptr16(const void*) { return 0; }

int main(int argc, char** argv) {
    if (argc < 4) return 2;
    const int n = atoi(argv[1]);
    FILE *f = fopen(argv[2], "rb"), *g = fopen(argv[3], "wb");
    if (!f || !g) return 1;
    std::vector<float> x(n);
    std::vector<double> med;
    std::vector<int> passes;
    while (fread(x.data(), 4, n, f) == (size_t)n) {
        std::vector<unsigned> key;
        int nv = 0;
        for (float v : x) {
            const bool ok = std::isfinite(v);
            key.push_back(ok ? key32(v) : BOX_NONE);
            nv += ok;
        }
        std::vector<unsigned> first(32, BOX_NONE);          // the kernel's sample: one warp's first keys
        for (int i = 0; i < 32 && i < n; i++) first[i] = key[i];
        std::sort(first.begin(), first.end());
        BoxBracket q;
        q.init(nv, first[9], first[22]);
        int it = 0;
        for (;; it++) {
            if (q.useful()) {
                int c = 0, d = 0;
                for (unsigned k : key) { c += k <= q.t; d += k <= q.u; }
                q.narrow(c, d);
            }
            if (q.done()) break;
            if (it > 100) { fprintf(stderr, "no end\n"); return 1; }
            q.next(it);
        }
        unsigned k1, k2;
        if (q.split) {
            k1 = 0u;
            k2 = BOX_NONE;
            for (unsigned k : key) {
                if (k <= q.cut) k1 = std::max(k1, k);
                else k2 = std::min(k2, k);
            }
        } else if (q.hi - q.lo == 1u) {
            k1 = k2 = q.hi;
        } else {
            std::vector<unsigned> left;
            for (unsigned k : key)
                if (q.holds(k)) left.push_back(k);
            if (left.size() > 32) { fprintf(stderr, "%zu left\n", left.size()); return 1; }
            std::sort(left.begin(), left.end());
            k1 = left[q.r1 - q.clo];
            k2 = left[q.r2 - q.clo];
        }
        med.push_back(median_of_keys(k1, k2));
        passes.push_back(it + 1);
    }
    fwrite(med.data(), 8, med.size(), g);
    fwrite(passes.data(), 4, passes.size(), g);
    fclose(f);
    fclose(g);
    return 0;
}
