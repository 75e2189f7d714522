// CPU driver of the register transforms (fft.cuh, proper.cu): the kernels' lane maps,
// twiddle slots and butterflies, lane by lane; the crossings through shared memory are
// the barrier.  usage:
//   host_fft_lanes full T dbl sign in out   (in, out: complex [n][T])
//   host_fft_lanes psf T ps in out          (in: f64 [n][ps]; out: complex128 [2][n][T], with the zeros left out of
//                                            the first two passes where the kernels do, and in none)
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <cmath>
#include <vector>
#include "proper.cu"

// library helpers the translation unit references (host driver only)
int argus_check_shape(const argus_shape&, size_t) { return 0; }
void argus_count_launch(int) {}
int argus_launch_status() { return 0; }

// a lane's twiddles read from the table (what TwReg holds in registers)
template <int T, typename C> struct HostTw {
    const C* tab;
    int lane;
    C get(int i) const { return tab[fft::tw_index<T>(i, lane)]; }
};

template <int T, int STEP, typename C> void cross_all(std::vector<C>& v, bool few) {
    std::vector<C> row(fft::Reg<T>::PT);
    for (int l = 0; l < T / 8; l++)
        for (int i = 0; i < 8; i++) row[fft::cross_to<T, STEP>(l, i)] = v[l * 8 + i];
    for (int l = 0; l < T / 8; l++)
        for (int m = 0; m < 8; m++)
            if (!few || m < 2 || m > 5) v[l * 8 + m] = row[fft::pad(l + m * (T / 8))];
            else v[l * 8 + m] = {NAN, NAN};                 // left out: not to be used
}

template <int T, int S, int STEP, bool FEW = false, typename C> void pass_all(std::vector<C>& v, const C* tab) {
    for (int l = 0; l < T / 8; l++) {
        C q[8];
        for (int m = 0; m < 8; m++) q[m] = v[l * 8 + m];
        fft::pass<T, S, STEP, FEW>(q, HostTw<T, C>{tab, l});
        for (int m = 0; m < 8; m++) v[l * 8 + m] = q[m];
    }
}

// the passes after the first
template <int T, int S, typename C> void tail(std::vector<C>& v, const C* tab, bool few) {
    cross_all<T, 0>(v, few);
    if (few) pass_all<T, S, 1, true>(v, tab);
    else pass_all<T, S, 1>(v, tab);
    cross_all<T, 1>(v, false);
    pass_all<T, S, 2>(v, tab);
    if constexpr (T == 1024) {
        cross_all<T, 2>(v, false);
        pass_all<T, S, 3>(v, tab);
    }
}

template <int T, typename C> void store(const std::vector<C>& v, FILE* f) {
    std::vector<C> o(T);
    for (int l = 0; l < T / 8; l++)
        for (int m = 0; m < 8; m++) o[l + m * (T / 8)] = v[l * 8 + m];
    fwrite(o.data(), sizeof(C), T, f);
}

template <int T, typename C> std::vector<C> table() {
    std::vector<C> t(T);
    for (int m = 0; m < T; m++) {
        const double a = 6.283185307179586476925286766559 * m / T;
        t[m].x = cos(a);
        t[m].y = -sin(a);
    }
    return t;
}

template <int T, int S, typename C> void full(FILE* f, FILE* g) {
    const std::vector<C> tab = table<T, C>();
    std::vector<C> x(T), v(T);
    while (fread(x.data(), sizeof(C), T, f) == T) {
        for (int l = 0; l < T / 8; l++) {
            C q[8];
            for (int m = 0; m < 8; m++) q[m] = x[l + m * (T / 8)];
            fft::dft8<S>(q);
            for (int m = 0; m < 8; m++) v[l * 8 + m] = q[m];
        }
        tail<T, S>(v, tab.data(), false);
        store<T>(v, g);
    }
}

template <int T> void psf(int ps, FILE* f, FILE* g) {
    const std::vector<double2> tab = table<T, double2>();
    std::vector<double> x(ps);
    std::vector<std::vector<double>> in;
    while (fread(x.data(), 8, ps, f) == (size_t)ps) in.push_back(x);
    for (int form = 0; form < 2; form++)
        for (const auto& p : in) {
            std::vector<double2> v(T);
            for (int l = 0; l < T / 8; l++) {
                bool any0 = false, any7 = false;            // over the lane's warp
                for (int w = l & ~31; w < (l & ~31) + 32 && w < T / 8; w++) {
                    any0 = any0 || psf_at<T>(ps, w, false) < ps;
                    any7 = any7 || psf_at<T>(ps, w, true) >= 0;
                }
                const int a = psf_at<T>(ps, l, false), b = psf_at<T>(ps, l, true);
                double2 q[8], v0 = {a < ps ? p[a] : 0.0, 0.0}, v7 = {b >= 0 ? p[b] : 0.0, 0.0};
                if (form == 0) {
                    psf_first(q, v0, v7, any0, any7);
                } else {
                    for (int m = 0; m < 8; m++) q[m] = {0.0, 0.0};
                    q[0] = v0;
                    q[7] = v7;
                    fft::dft8<-1>(q);
                }
                for (int m = 0; m < 8; m++) v[l * 8 + m] = q[m];
            }
            tail<T, -1>(v, tab.data(), form == 0 && psf_few<T>(ps));
            store<T>(v, g);
        }
}

int main(int argc, char** argv) {
    if (argc < 6) return 2;
    const bool whole = !strcmp(argv[1], "full");
    const int T = atoi(argv[2]), a = atoi(argv[3]), sign = whole ? atoi(argv[4]) : 0;
    FILE *f = fopen(argv[whole ? 5 : 4], "rb"), *g = fopen(argv[whole ? 6 : 5], "wb");
    if (!f || !g) return 1;
    const auto run = [&](auto t) {
        constexpr int N = decltype(t)::value;
        if (!whole) psf<N>(a, f, g);
        else if (a && sign < 0) full<N, -1, double2>(f, g);
        else if (a) full<N, 1, double2>(f, g);
        else if (sign < 0) full<N, -1, float2>(f, g);
        else full<N, 1, float2>(f, g);
    };
    if (T == 256) run(std::integral_constant<int, 256>{});
    else if (T == 512) run(std::integral_constant<int, 512>{});
    else run(std::integral_constant<int, 1024>{});
    fclose(f);
    fclose(g);
    return 0;
}
