// Proper-image statistics on square tiles: ZOGY subtraction (below) and the
// proper coadd (after it) share one plan and the register FFTs of fft.cuh.
//
// Both are sums of real images filtered by kernels with real images, and two real images
// ride one complex row transform, Z = DFT[N + i R].
//
// ZOGY proper image subtraction (paper Sec. 4.2: ZOGY at base cadence and in
// deep coadds; the statistic of Zackay, Ofek & Gal-Yam 2016), per T x T tile:
//   1. psf_rows / psf_cols (new PSFs only): FP64 transforms of the stamps, placed
//      with their centre at (0, 0) (wrapping around), each real PSF on the half
//      plane kx <= T/2; (Pn, Pr) kept in FP32, max(|Pn|^2, |Pr|^2) also in FP64;
//   2. row_fwd: rows of N + i R;
//   3. zogy_col: a column and its mirror per thread: both forward, the images
//      separated (N^ = (Z(k) + conj Z(-k)) / 2), and per frequency of the half plane
//        den = sqrt(sn^2 Fr^2 |Pr|^2 + sr^2 Fn^2 |Pn|^2)
//        D   = (Fr Pr N - Fn Pn R) / den
//        P_D = Fr Fn Pr Pn / (F_D den),   F_D = Fr Fn / sqrt(sn^2 Fr^2 + sr^2 Fn^2)
//        S   = F_D D conj(P_D)
//      all 0 where max(|Pn|, |Pr|) < eps (decided in FP64; below that floor the
//      PSF transforms are rounding), inverse columns of each, and sum |P_D|^2 per
//      tile, which gives sigma_S = F_D ||P_D||_2;
//   4. row_inv_real: rows of D + i S (and of P_D when asked for), divided by T^2.
// D is small where N and R agree, so the images are separated before the quotient: with
// D left in one product with Z, its inverse columns carry the larger sum of the images
// too, and D's error was 1.25 times as large.  S has an inverse column of its own, free of
// D's rounding.  The PSF transforms are FP64 so that the floor decisions and the small
// transforms near it are those of an FP64 reference; the images and the
// filters are FP32.  216 tiles of 512^2 with a PSF pair each: 3.35 ms, against
// 12.9 ms with whole FP64 2-D transforms and a combine pass over mirrored pairs.
#include "argus_internal.cuh"
#include "fft.cuh"

#include <cmath>
#include <cstdlib>

struct argus_proper_plan {
    int device;
    int tile;
    int max_tiles;
    int psf_tiles;          // ZOGY PSF transforms the plan holds: that many tiles', -1 one shared pair, 0 none
    unsigned char* pool;    // pool_bytes() of scratch: see zogy_layout and run_coadd
    double* psd;            // [max_tiles][zogy_blocks] partial sums of |P_D(k)|^2
    float2* tw32;           // [T] e^{-2 pi i m / T}
    double2* tw64;
};

namespace {

// 48 bytes per tile pixel, and 64 per pixel of one tile more so that a coadd of a
// small plan still holds a few frame pairs at a time.
size_t pool_bytes(int tile, int max_tiles) { return ((size_t)max_tiles * 48 + 64) * (size_t)tile * tile; }

__host__ __device__ __forceinline__ float2 f2(double2 v) { return make_float2((float)v.x, (float)v.y); }

// ---------------------------------------------------------------------------
// Tiles between the row and the column passes lie in blocks of CB columns,
// [tile][T / CB][T rows][CB], so that a column CTA reads one contiguous block.
template <int T> __device__ __forceinline__ int blocked(int y, int x) {
    constexpr int CB = fft::Reg<T>::CB;
    return ((x / CB) * T + y) * CB + x % CB;
}

constexpr int ROW_ITER = 4;   // row groups of a row CTA (its twiddles are loaded once)

// Resident CTAs asked for: 128 registers a thread hold the eight values, the twiddles
// and a filter's or a mirror's loads without spills (three CTAs of 256 spill).
template <int T> constexpr int min_ctas() { return T == 1024 ? 1 : 2; }

struct RowArgs {
    const float* s0;        // first image of pair 0; pair p's at s0 + p * pair_stride
    const float* s1;        // second image
    long pair_stride;
    int n_second;           // pairs that have a second image
    long pitch;
    int w, h;
    const int* org;         // tile origins: (x, y) at org + t * org_stride
    int org_stride;
    int n_tiles;
    const float2* tw;
    float2* z;              // [pair][tile] blocked
};

// Forward rows of image pairs, straight from the frames (pixels off the frame
// are 0).  Grid (tiles * T / (CB ROW_ITER), pairs).
template <int T>
__global__ void __launch_bounds__(fft::Reg<T>::THREADS, min_ctas<T>()) row_fwd_kernel(RowArgs a) {
    using Rg = fft::Reg<T>;
    extern __shared__ __align__(16) unsigned char fft_smem[];
    float2* sm = reinterpret_cast<float2*>(fft_smem);
    constexpr int PER = T / (Rg::CB * ROW_ITER);
    const int lane = threadIdx.x % Rg::LANES, seq = threadIdx.x / Rg::LANES;
    const int t = blockIdx.x / PER, y0 = (blockIdx.x - t * PER) * Rg::CB * ROW_ITER, p = blockIdx.y;
    const int ox = a.org[(long)t * a.org_stride], oy = a.org[(long)t * a.org_stride + 1];
    const float* s0 = a.s0 + p * a.pair_stride;
    const float* s1 = p < a.n_second ? a.s1 + p * a.pair_stride : nullptr;
    float2* z = a.z + ((long)p * a.n_tiles + t) * T * T;
    const fft::TwReg<T> tw(a.tw, lane);
    float2* b0 = sm + seq * Rg::PT;
    float2* b1 = sm + (Rg::CB + seq) * Rg::PT;
    float2 v[8], nx[8];
    // row y of the pair (the next group's row is loaded while this one is transformed)
    const auto load = [&](int y, float2 (&d)[8]) {
        const int gy = oy + y;
        const bool row = gy >= 0 && gy < a.h;
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const int gx = ox + lane + m * Rg::LANES;
            const bool in = row && gx >= 0 && gx < a.w;
            const long q = (long)gy * a.pitch + gx;
            d[m].x = in ? __ldg(s0 + q) : 0.0f;
            d[m].y = in && s1 ? __ldg(s1 + q) : 0.0f;
        }
    };
    load(y0 + seq, nx);
#pragma unroll 1
    for (int i = 0; i < ROW_ITER; i++) {
        const int y = y0 + i * Rg::CB + seq;
#pragma unroll
        for (int m = 0; m < 8; m++) v[m] = nx[m];
        if (i + 1 < ROW_ITER) load(y + Rg::CB, nx);
        fft::fft_reg<T, -1, 1>(v, tw, b0, b1, lane);
#pragma unroll
        for (int m = 0; m < 8; m++) z[blocked<T>(y, lane + m * Rg::LANES)] = v[m];
    }
}

// Inverse rows of x (and of y, when given): out_x = Re IDFT[x] / T^2 per row, out_y
// likewise.  W = X + i Y of the conjugate-symmetric parts X(k) = (x(k) +
// conj x(-k)) / 2, so one transform gives both.  Grid tiles * T / (CB ROW_ITER).
template <int T>
__global__ void __launch_bounds__(fft::Reg<T>::THREADS, min_ctas<T>()) row_inv_kernel(const float2* x, const float2* y, float* out_x,
                                                                      float* out_y, const float2* twg) {
    using Rg = fft::Reg<T>;
    extern __shared__ __align__(16) unsigned char fft_smem[];
    float2* sm = reinterpret_cast<float2*>(fft_smem);
    constexpr int PER = T / (Rg::CB * ROW_ITER);
    const int lane = threadIdx.x % Rg::LANES, seq = threadIdx.x / Rg::LANES;
    const int t = blockIdx.x / PER, y0 = (blockIdx.x - t * PER) * Rg::CB * ROW_ITER;
    const long base = (long)t * T * T;
    x += base;
    if (y) y += base;
    const fft::TwReg<T> tw(twg, lane);
    float2* b0 = sm + seq * Rg::PT;
    float2* b1 = sm + (Rg::CB + seq) * Rg::PT;
    const float half = 0.5f / ((float)T * (float)T);           // a power of two: exact
#pragma unroll 1
    for (int i = 0; i < ROW_ITER; i++) {
        const int r = y0 + i * Rg::CB + seq;
        float2 v[8];
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const int k = lane + m * Rg::LANES, q = blocked<T>(r, k), n = blocked<T>(r, (T - k) & (T - 1));
            const float2 p = x[q], pc = x[n];
            v[m] = make_float2(p.x + pc.x, p.y - pc.y);
            if (y) {
                const float2 s = y[q], sc = y[n];
                v[m].x -= s.y - sc.y;
                v[m].y += s.x + sc.x;
            }
        }
        fft::fft_reg<T, 1, 1>(v, tw, b0, b1, lane);
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const long e = base + (long)r * T + lane + m * Rg::LANES;
            out_x[e] = v[m].x * half;
            if (y) out_y[e] = v[m].y * half;
        }
    }
}

// Inverse rows of tiles whose half-inverted columns are those of real images (X(-k) = conj
// X(k)): TWO, X in the columns 0 < kx < T/2 and Y in their mirrors' places, X + i Y in
// columns 0 and T/2 (where both are real), and one transform gives both; otherwise X alone in
// the columns up to T/2.  Grid tiles * T / (CB ROW_ITER).
template <int T, bool TWO>
__global__ void __launch_bounds__(fft::Reg<T>::THREADS, min_ctas<T>()) row_inv_real_kernel(const float2* z, float* out_x, float* out_y,
                                                                          const float2* twg) {
    using Rg = fft::Reg<T>;
    extern __shared__ __align__(16) unsigned char fft_smem[];
    float2* sm = reinterpret_cast<float2*>(fft_smem);
    constexpr int PER = T / (Rg::CB * ROW_ITER);
    const int lane = threadIdx.x % Rg::LANES, seq = threadIdx.x / Rg::LANES;
    const int t = blockIdx.x / PER, y0 = (blockIdx.x - t * PER) * Rg::CB * ROW_ITER;
    const long base = (long)t * T * T;
    z += base;
    const fft::TwReg<T> tw(twg, lane);
    float2* b0 = sm + seq * Rg::PT;
    float2* b1 = sm + (Rg::CB + seq) * Rg::PT;
    const float scale = 1.0f / ((float)T * (float)T);          // a power of two: exact
#pragma unroll 1
    for (int i = 0; i < ROW_ITER; i++) {
        const int r = y0 + i * Rg::CB + seq;
        float2 v[8];
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const int k = lane + m * Rg::LANES;                // k < T/2 where m < 4
            const float2 p = z[blocked<T>(r, k)], n = z[blocked<T>(r, (T - k) & (T - 1))];
            if (lane == 0 && m % 4 == 0) v[m] = p;
            else if (TWO) v[m] = m < 4 ? make_float2(p.x - n.y, p.y + n.x) : make_float2(n.x + p.y, p.x - n.y);
            else v[m] = m < 4 ? p : fft::cconj(n);
        }
        fft::fft_reg<T, 1, 1>(v, tw, b0, b1, lane);
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const long e = base + (long)r * T + lane + m * Rg::LANES;
            out_x[e] = v[m].x * scale;
            if (TWO) out_y[e] = v[m].y * scale;
        }
    }
}

// ---------------------------------------------------------------------------
// PSF transforms (FP64).  A stamp fills at most 63 of a tile's rows: only those
// rows are transformed, and the first radix-8 pass of a sequence has at most two
// nonzero inputs per lane (position lane and position lane + 7 T/8), which leaves
// rotations by multiples of 45 degrees and two passes.  Each real PSF takes the
// half plane kx <= T/2.  On 216 tiles of 512^2 the FP64 pipe (2 FMA per clock per
// SM) bounds them.
struct PsfArgs {
    const float* p0;        // first stamp of (tile 0, pair 0); tile t's pair p at p0 + t * tile_stride + p * pair_stride
    const float* p1;        // second stamp
    long tile_stride, pair_stride;
    int n_second;           // pairs that have a second stamp
    int n_pairs;
    int ps;
    const double2* tw;
    double2* rows;          // [tile][pair][2][ps][T / 2 + 1]
};

// First pass of a sequence with values only at positions lane (v0; none in any lane of the
// warp unless any0) and lane + 7 T/8 (v7, any7).  Most warps hold values of one kind at
// most, which need no sums (column transforms of 31 x 31 stamps in 216 tiles of 512: 2.45 ->
// 2.25 ms).
__host__ __device__ __forceinline__ void psf_first(double2 (&v)[8], double2 v0, double2 v7, bool any0, bool any7) {
    const double r = 0.70710678118654752440;
    if (!any7) {
#pragma unroll
        for (int m = 0; m < 8; m++) v[m] = v0;
        return;
    }
    const double2 d1 = make_double2(r * (v7.x - v7.y), r * (v7.x + v7.y));    // v7 e^{i pi / 4}
    const double2 d3 = make_double2(-d1.y, d1.x);                             // v7 e^{3 i pi / 4}
    const double2 d2 = make_double2(-v7.y, v7.x);
    if (!any0) {
        v[0] = v7; v[4] = make_double2(-v7.x, -v7.y);
        v[1] = d1; v[5] = make_double2(-d1.x, -d1.y);
        v[2] = d2; v[6] = make_double2(-d2.x, -d2.y);
        v[3] = d3; v[7] = make_double2(-d3.x, -d3.y);
        return;
    }
    v[0] = fft::cadd(v0, v7); v[4] = fft::csub(v0, v7);
    v[1] = fft::cadd(v0, d1); v[5] = fft::csub(v0, d1);
    v[2] = fft::cadd(v0, d2); v[6] = fft::csub(v0, d2);
    v[3] = fft::cadd(v0, d3); v[7] = fft::csub(v0, d3);
}

// The stamp pixels at positions lane and lane - T/8 of a sequence, its centre at 0; none where
// not in [0, ps).
template <int T> __host__ __device__ __forceinline__ int psf_at(int ps, int lane, bool wrapped) {
    return ps / 2 + lane - (wrapped ? T / 8 : 0);
}

constexpr int PSEQ = 2;       // FP64 sequences per CTA

// The other passes of a stamp's sequence.  A stamp of half-side below T/32 leaves half of
// the second pass's values zero too: FP64 arithmetic bounds these kernels, and its radix-8
// butterflies then take 52 operations instead of 84 (column transforms of 31 x 31 stamps
// in 216 tiles of 512: 2.87 -> 2.45 ms).
template <int T> __host__ __device__ __forceinline__ bool psf_few(int ps) {
    return T == 1024 || ps / 2 < T / 32;                   // (a side is at most 63)
}
template <int T, int ST>
__device__ __forceinline__ void psf_tail(double2 (&v)[8], int ps, const fft::TwTab<T>& tw, double2*& b0, double2*& b1, int lane) {
    if (psf_few<T>(ps)) fft::fft_tail<T, -1, ST, true>(v, tw, b0, b1, lane);
    else fft::fft_tail<T, -1, ST>(v, tw, b0, b1, lane);
}

// Row transforms of a pair's stamps (z = p0 + i p1, separated within the row).
// Grid psf_tiles * n_pairs * ceil(ps / PSEQ).
template <int T>
__global__ void __launch_bounds__(PSEQ * fft::Reg<T>::LANES) psf_rows_kernel(PsfArgs a) {
    using Rg = fft::Reg<T>;
    extern __shared__ __align__(16) unsigned char fft_smem[];
    double2* sm = reinterpret_cast<double2*>(fft_smem);
    const int lane = threadIdx.x % Rg::LANES, seq = threadIdx.x / Rg::LANES;
    const int nb = (a.ps + PSEQ - 1) / PSEQ;
    const long tp = blockIdx.x / nb;                        // tile * n_pairs + pair
    const int row = (int)(blockIdx.x - tp * nb) * PSEQ + seq;
    const long t = tp / a.n_pairs;
    const int p = (int)(tp - t * a.n_pairs);
    const bool live = row < a.ps;
    const long o = t * a.tile_stride + p * a.pair_stride + (long)row * a.ps;
    const bool two = p < a.n_second;
    const int q = psf_at<T>(a.ps, lane, false), u = psf_at<T>(a.ps, lane, true);
    double2 v0 = make_double2(0.0, 0.0), v7 = v0, v[8];
    if (live && q < a.ps) {
        v0.x = a.p0[o + q];
        if (two) v0.y = a.p1[o + q];
    }
    if (live && u >= 0) {
        v7.x = a.p0[o + u];
        if (two) v7.y = a.p1[o + u];
    }
    psf_first(v, v0, v7, __any_sync(0xffffffffu, q < a.ps), __any_sync(0xffffffffu, u >= 0));
    double2* b0 = sm + seq * Rg::PT;
    double2* b1 = sm + (PSEQ + seq) * Rg::PT;
    const fft::TwTab<T> tw{a.tw, lane};
    psf_tail<T, 1>(v, a.ps, tw, b0, b1, lane);
#pragma unroll
    for (int m = 0; m < 8; m++) b0[lane + m * Rg::LANES] = v[m];
    __syncthreads();
    if (!live) return;
    constexpr int HW = T / 2 + 1;
    double2* d0 = a.rows + (tp * 2 * a.ps + row) * HW;
    double2* d1 = d0 + (long)a.ps * HW;
    for (int k = lane; k < HW; k += Rg::LANES) {
        const double2 A = b0[k], B = b0[(T - k) & (T - 1)];
        d0[k] = make_double2(0.5 * (A.x + B.x), 0.5 * (A.y - B.y));
        d1[k] = make_double2(0.5 * (A.y + B.y), -0.5 * (A.x - B.x));
    }
}

// Column kx of one stamp's row transforms (rows: that stamp's [ps][T / 2 + 1]).
template <int T>
__device__ __forceinline__ void psf_column(double2 (&v)[8], const double2* rows, int ps, int kx, const fft::TwTab<T>& tw,
                                           double2*& b0, double2*& b1, int lane) {
    constexpr int HW = T / 2 + 1;
    const int q = psf_at<T>(ps, lane, false), u = psf_at<T>(ps, lane, true);
    double2 v0 = make_double2(0.0, 0.0), v7 = v0;
    if (kx < HW && q < ps) v0 = rows[(long)q * HW + kx];
    if (kx < HW && u >= 0) v7 = rows[(long)u * HW + kx];
    psf_first(v, v0, v7, __any_sync(0xffffffffu, q < ps), __any_sync(0xffffffffu, u >= 0));
    psf_tail<T, PSEQ>(v, ps, tw, b0, b1, lane);
}

// ---------------------------------------------------------------------------
// ZOGY

struct ZArgs {
    const argus_zogy_tile* tiles;
    int n_tiles;
    int psf_tiles;            // tiles with their own PSF pair: n_tiles, or 1 when all share one
    double eps2;
    float lo2, hi2;           // below lo2 certainly under the floor, above hi2 certainly not
    const float4* spec;       // [psf tile][T / 2 + 1][T] (Pn, Pr) at (kx, ky)
    const double* top2;       // [psf tile][T / 2 + 1][T] max(|Pn|^2, |Pr|^2)
    float2* z;                // rows of N + i R in; half-inverted D, S out (the form row_inv_real takes)
    float2* zp;               // half-inverted P_D in columns up to T/2, or null
    double* psd;              // [tile][zogy_blocks]
    const float2* tw;
    double* sigma_S;
};

__host__ __device__ __forceinline__ float zogy_FD(argus_zogy_tile tp) {
    return tp.Fr * tp.Fn / sqrtf(tp.sn * tp.sn * tp.Fr * tp.Fr + tp.sr * tp.sr * tp.Fn * tp.Fn);
}

// D, S and P_D at one frequency k from A = Z(k) and B = Z(-k), Z = DFT[N + i R], and the PSFs'
// transforms there; 0 under the floor (above = false).  Host-callable, so a CPU driver can run
// the same code.
__host__ __device__ __forceinline__ void zogy_point(float2 A, float2 B, float2 pn, float2 pr, bool above, argus_zogy_tile tp,
                                                      float FD, float2& Dh, float2& Sh, float2& PD) {
    // N = (A + conj B) / 2, R = (A - conj B) / 2i
    const float2 Nh = make_float2(0.5f * (A.x + B.x), 0.5f * (A.y - B.y));
    const float2 Rh = make_float2(0.5f * (A.y + B.y), -0.5f * (A.x - B.x));
    const float Fn = tp.Fn, Fr = tp.Fr, sn = tp.sn, sr = tp.sr;
    const float den = sqrtf(sn * sn * Fr * Fr * (pr.x * pr.x + pr.y * pr.y) +
                            sr * sr * Fn * Fn * (pn.x * pn.x + pn.y * pn.y));
    Dh = PD = make_float2(0.0f, 0.0f);
    if (above && den > 0.0f) {
        // Fr Pr N - Fn Pn R
        const float2 u = make_float2(Fr * (pr.x * Nh.x - pr.y * Nh.y) - Fn * (pn.x * Rh.x - pn.y * Rh.y),
                                     Fr * (pr.x * Nh.y + pr.y * Nh.x) - Fn * (pn.x * Rh.y + pn.y * Rh.x));
        Dh = make_float2(u.x / den, u.y / den);
        const float g = Fr * Fn / (FD * den);
        PD = make_float2(g * (pr.x * pn.x - pr.y * pn.y), g * (pr.x * pn.y + pr.y * pn.x));
    }
    Sh = make_float2(FD * (Dh.x * PD.x + Dh.y * PD.y), FD * (Dh.y * PD.x - Dh.x * PD.y));
}

// X + i Y, and its value at -k for X, Y the transforms of real images.
__host__ __device__ __forceinline__ float2 plus_i(float2 X, float2 Y) { return make_float2(X.x - Y.y, X.y + Y.x); }
__host__ __device__ __forceinline__ float2 plus_i_mirror(float2 X, float2 Y) { return make_float2(X.x + Y.y, Y.x - X.y); }

// The step of one frequency pair on whole transforms, C = z2(k), E = z2(-k) with z2 = DFT[Pn + i
// Pr]: W(k) = D + i S and W(-k), P_D(k); returns |P_D(k)|^2 (the CPU driver's form).
[[maybe_unused]] __host__ __device__ __forceinline__ void zogy_pair(float2 A, float2 B, double2 C, double2 E, argus_zogy_tile tp,
                                                   double eps2, float2& Wq, float2& Wp, float2& PD, double& p2) {
    const double2 Pn = make_double2(0.5 * (C.x + E.x), 0.5 * (C.y - E.y));
    const double2 Pr = make_double2(0.5 * (C.y + E.y), -0.5 * (C.x - E.x));
    const double mn = Pn.x * Pn.x + Pn.y * Pn.y, mr = Pr.x * Pr.x + Pr.y * Pr.y;
    float2 Dh, Sh;
    zogy_point(A, B, f2(Pn), f2(Pr), mn >= eps2 || mr >= eps2, tp, zogy_FD(tp), Dh, Sh, PD);
    p2 = (double)PD.x * PD.x + (double)PD.y * PD.y;
    Wq = plus_i(Dh, Sh);
    Wp = plus_i_mirror(Dh, Sh);
}

// Grid psf_tiles * ceil((T / 2 + 1) / PSEQ).
template <int T>
__global__ void __launch_bounds__(PSEQ * fft::Reg<T>::LANES) zogy_psf_cols_kernel(PsfArgs a, float4* spec,
                                                                                 double* top2) {
    using Rg = fft::Reg<T>;
    extern __shared__ __align__(16) unsigned char fft_smem[];
    double2* sm = reinterpret_cast<double2*>(fft_smem);
    constexpr int HW = T / 2 + 1, NB = (HW + PSEQ - 1) / PSEQ;
    const int c = threadIdx.x % PSEQ, lane = threadIdx.x / PSEQ;
    const long t = blockIdx.x / NB;
    const int kx = (int)(blockIdx.x - t * NB) * PSEQ + c;
    double2* b0 = sm + c;
    double2* b1 = sm + PSEQ * Rg::PT + c;
    const fft::TwTab<T> tw{a.tw, lane};
    const double2* rows = a.rows + t * 2 * a.ps * HW;
    double2 v[8];
    float2 pn[8];
    double mn[8];
    psf_column<T>(v, rows, a.ps, kx, tw, b0, b1, lane);
#pragma unroll
    for (int m = 0; m < 8; m++) {
        pn[m] = f2(v[m]);
        mn[m] = v[m].x * v[m].x + v[m].y * v[m].y;
    }
    psf_column<T>(v, rows + (long)a.ps * HW, a.ps, kx, tw, b0, b1, lane);
    if (kx >= HW) return;
#pragma unroll
    for (int m = 0; m < 8; m++) {
        const double mr = v[m].x * v[m].x + v[m].y * v[m].y;
        const float2 pr = f2(v[m]);
        const long e = (t * HW + kx) * T + lane + m * Rg::LANES;
        spec[e] = make_float4(pn[m].x, pn[m].y, pr.x, pr.y);
        top2[e] = mn[m] > mr ? mn[m] : mr;                 // NaN fails every comparison with the floor, as its parts do
    }
}

// Columns of the tiles: forward, quotient, inverse.  A thread takes column kx and its mirror
// T - kx (columns 0 and T/2, each its own mirror, alone); after the forward transforms the
// mirror crosses through shared memory, as Z(-k) lies in it at -ky.  The two sequences go
// through a transform side by side.  sum |P_D|^2: a thread's 16 exact squares as an unevaluated
// FP32 pair (at most 2^-44 of it off), FP64 over the threads; sigma_S's error against 64 bits, 3e-8 to
// 6e-8 from P_D in FP32, is that of FP64 sums, which cost 0.1 ms (two operations per clock and
// SM).  Its loads bound it with the 16 warps an SM that 128 registers leave.  216 tiles of
// 512 with kept PSFs, the whole call: 0.91 ms; with a column per thread, twice as many inverse
// transforms and stores, 1.39.  Grid n_tiles * zogy_blocks<T>().
template <int T> __host__ __device__ constexpr int zogy_blocks() { return T / (2 * fft::Reg<T>::CB) + 1; }

template <int T>
__global__ void __launch_bounds__(fft::Reg<T>::THREADS, min_ctas<T>()) zogy_col_kernel(ZArgs a) {
    using Rg = fft::Reg<T>;
    constexpr int CB = Rg::CB, L = Rg::LANES, NB = zogy_blocks<T>(), HW = T / 2 + 1;
    extern __shared__ __align__(16) unsigned char fft_smem[];
    float2* sm = reinterpret_cast<float2*>(fft_smem);
    __shared__ double red[Rg::THREADS / 32];
    const int c = threadIdx.x % CB, lane = threadIdx.x / CB;
    const int t = blockIdx.x / NB, xb = blockIdx.x - t * NB, kx = xb * CB + c;
    const bool live = kx <= T / 2, self = kx == 0 || kx == T / 2;
    float2* zk = a.z + (long)t * T * T + blocked<T>(lane, live ? kx : 0);
    float2* zm = a.z + (long)t * T * T + blocked<T>(lane, live && !self ? T - kx : 0);
    const fft::TwReg<T> tw(a.tw, lane);
    float2* v0 = sm + c;                                   // two buffers for each of the two sequences
    float2* v1 = v0 + CB * Rg::PT;
    float2* w0 = v1 + CB * Rg::PT;
    float2* w1 = w0 + CB * Rg::PT;
    const argus_zogy_tile tp = a.tiles[t];
    const float FD = zogy_FD(tp);
    const long sp = ((a.psf_tiles == 1 ? 0L : (long)t) * HW + (live ? kx : 0)) * T + lane;
    float2 v[8], w[8], P[8];
#pragma unroll
    for (int m = 0; m < 8; m++) w[m] = live && !self ? zm[m * L * CB] : make_float2(0.0f, 0.0f);
#pragma unroll
    for (int m = 0; m < 8; m++) v[m] = live ? zk[m * L * CB] : make_float2(0.0f, 0.0f);
    // the PSF transforms are wanted after these: on their way to the L2 now (registers leave no
    // room to load them ahead)
    if (lane % 8 == 0) {
#pragma unroll
        for (int m = 0; m < 8; m++) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.spec + sp + m * L));
    }
    fft::fft_reg2<T, -1, CB>(v, w, tw, v0, v1, w0, w1, lane);
#pragma unroll
    for (int m = 0; m < 8; m++) w0[fft::pad(lane + m * L) * CB] = self ? v[m] : w[m];
    __syncthreads();
    float hs = 0.0f, ls = 0.0f;
#pragma unroll
    for (int m = 0; m < 8; m++) {
        const float4 q = __ldg(a.spec + sp + m * L);
        const float2 pn = make_float2(q.x, q.y), pr = make_float2(q.z, q.w);
        // the floor: FP32 moduli decide except next to it, where the FP64 one does
        const float m2 = fmaxf(pn.x * pn.x + pn.y * pn.y, pr.x * pr.x + pr.y * pr.y);
        bool above = m2 > a.hi2;
        if (!above && !(m2 < a.lo2)) above = __ldg(a.top2 + sp + m * L) >= a.eps2;
        float2 D;
        zogy_point(v[m], w0[fft::pad((T - lane - m * L) & (T - 1)) * CB], pn, pr, above, tp, FD, D, w[m], P[m]);
        v[m] = self ? plus_i(D, w[m]) : D;                 // columns 0 and T/2: X + i Y, whose inverse is real and real
#pragma unroll
        for (int i = 0; i < 2; i++) {                      // exact square, two-sum into the pair
            const float d = i ? P[m].y : P[m].x, h = d * d, e2 = fmaf(d, d, -h), n = hs + h, b = n - hs;
            ls += e2 + ((hs - (n - b)) + (h - b));
            hs = n;
        }
    }
    double psd = live ? ((double)hs + (double)ls) * (self ? 1.0 : 2.0) : 0.0;      // k and -k
    for (int o = 16; o > 0; o >>= 1) psd += __shfl_xor_sync(0xffffffffu, psd, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = psd;
    // (barriers: red is complete after it, and w0 is read before it is written)
    fft::fft_reg2<T, 1, CB>(v, w, tw, v1, v0, w1, w0, lane);
#pragma unroll
    for (int m = 0; m < 8; m++) {
        if (live) zk[m * L * CB] = v[m];
        if (live && !self) zm[m * L * CB] = w[m];
    }
    if (a.zp) {
        fft::fft_reg<T, 1, CB>(P, tw, v1, v0, lane);
#pragma unroll
        for (int m = 0; m < 8; m++)
            if (live) a.zp[zk - a.z + m * L * CB] = P[m];
    }
    if (threadIdx.x == 0) {
        double r = 0.0;
        for (int i = 0; i < Rg::THREADS / 32; i++) r += red[i];
        a.psd[(long)t * NB + xb] = r;
    }
}

template <int T>
__global__ void zogy_sigma_kernel(ZArgs a) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.n_tiles) return;
    constexpr int NB = zogy_blocks<T>();
    const argus_zogy_tile tp = a.tiles[t];
    const double Fn = tp.Fn, Fr = tp.Fr, sn = tp.sn, sr = tp.sr;
    const double FD = Fr * Fn / sqrt(sn * sn * Fr * Fr + sr * sr * Fn * Fn);
    double s = 0.0;
    for (int i = 0; i < NB; i++) s += a.psd[(long)t * NB + i];
    a.sigma_S[t] = FD * sqrt(s / ((double)T * T));
}

template <int T> constexpr size_t img_smem() { return 2 * (size_t)fft::Reg<T>::CB * fft::Reg<T>::PT * sizeof(float2); }

template <int T>
void launch_rows(const RowArgs& r, int pairs, cudaStream_t s) {
    const unsigned gx = (unsigned)((long)r.n_tiles * (T / (fft::Reg<T>::CB * ROW_ITER)));
    row_fwd_kernel<T><<<dim3(gx, pairs), fft::Reg<T>::THREADS, img_smem<T>(), s>>>(r);
    argus_count_launch(1);
}

template <int T>
void launch_inv(const float2* x, const float2* y, float* ox, float* oy, int n, const float2* tw, cudaStream_t s) {
    const unsigned gx = (unsigned)((long)n * (T / (fft::Reg<T>::CB * ROW_ITER)));
    row_inv_kernel<T><<<gx, fft::Reg<T>::THREADS, img_smem<T>(), s>>>(x, y, ox, oy, tw);
    argus_count_launch(1);
}

template <int T>
void launch_inv_real(const float2* z, float* ox, float* oy, int n, const float2* tw, cudaStream_t s) {
    const unsigned gx = (unsigned)((long)n * (T / (fft::Reg<T>::CB * ROW_ITER)));
    if (oy) row_inv_real_kernel<T, true><<<gx, fft::Reg<T>::THREADS, img_smem<T>(), s>>>(z, ox, oy, tw);
    else row_inv_real_kernel<T, false><<<gx, fft::Reg<T>::THREADS, img_smem<T>(), s>>>(z, ox, nullptr, tw);
    argus_count_launch(1);
}

template <int T> constexpr size_t psf_smem() { return 2 * PSEQ * (size_t)fft::Reg<T>::PT * sizeof(double2); }
template <int T> constexpr unsigned psf_col_blocks() { return (T / 2 + 1 + PSEQ - 1) / PSEQ; }

template <int T>
int run(argus_proper_plan* p, ZArgs& a, const RowArgs& rows, const PsfArgs* psf, float* D, float* S, float* PD,
        cudaStream_t s) {
    using Rg = fft::Reg<T>;
    // the pool, in bytes per pixel of max_tiles tiles: z 8, P_D 8, (spec, top2) 16 -- kept for
    // calls that reuse the PSFs -- and 16 for the PSFs' row transforms
    const size_t N = (size_t)p->max_tiles * T * T, half = (size_t)(T / 2 + 1) * T;
    a.z = reinterpret_cast<float2*>(p->pool);
    a.zp = PD ? reinterpret_cast<float2*>(p->pool + 8 * N) : nullptr;
    float4* spec = reinterpret_cast<float4*>(p->pool + 16 * N);
    double* top2 = reinterpret_cast<double*>(spec + half * p->max_tiles);
    a.spec = spec;
    a.top2 = top2;
    a.psd = p->psd;
    a.tw = p->tw32;
    if (psf) {
        PsfArgs q = *psf;
        q.tw = p->tw64;
        q.rows = reinterpret_cast<double2*>(p->pool + 32 * N);
        psf_rows_kernel<T><<<(unsigned)((long)a.psf_tiles * ((q.ps + PSEQ - 1) / PSEQ)), PSEQ * Rg::LANES, psf_smem<T>(), s>>>(q);
        zogy_psf_cols_kernel<T><<<(unsigned)a.psf_tiles * psf_col_blocks<T>(), PSEQ * Rg::LANES, psf_smem<T>(), s>>>(q, spec, top2);
        argus_count_launch(2);
    }
    RowArgs r = rows;
    r.tw = p->tw32;
    r.z = a.z;
    launch_rows<T>(r, 1, s);
    zogy_col_kernel<T><<<(unsigned)a.n_tiles * zogy_blocks<T>(), Rg::THREADS, 2 * img_smem<T>(), s>>>(a);
    argus_count_launch(1);
    launch_inv_real<T>(a.z, D, S, a.n_tiles, p->tw32, s);
    if (PD) launch_inv_real<T>(a.zp, PD, nullptr, a.n_tiles, p->tw32, s);
    if (a.sigma_S) {
        zogy_sigma_kernel<T><<<(a.n_tiles + 127) / 128, 128, 0, s>>>(a);
        argus_count_launch(1);
    }
    return argus_launch_status();
}

// ---------------------------------------------------------------------------
// Proper coaddition (paper Sec. 4.1.3: a per-image matched filter; the
// statistic of Zackay & Ofek 2017).  The frames of a pair are never separated: with Z =
// DFT[M_0 + i M_1] and c_0, c_1 transforms of real kernels,
//   Re IDFT[(c_0 - i c_1) Z] = IDFT[c_0 M_0^ + c_1 M_1^]
// (the other two products' inverses are imaginary), so a pair costs one complex product per
// frequency and the real parts are taken by the inverse rows.  With w_j = F_j / s_j^2:
//   S = sum_j IDFT[w_j conj(P_j) M_j] = Re IDFT[U],
//   U = sum over frame pairs of (w_0 conj P_0 - i w_1 conj P_1) DFT[M_0 + i M_1]
// (FP32), den^2 = sum_j F_j^2 / s_j^2 |P_j|^2 and max_j |P_j|^2 in FP64 on the half
// plane.  Then R = Re IDFT[U / den] (0 below the frequency floor) and P_R =
// IDFT[den / F_R], F_R = sqrt(sum_j F_j^2 / s_j^2).
// The column kernel keeps U of its columns in registers while it walks the frame
// pairs, so a pair costs one write and one read of its row transforms: 30 frames
// of 216 512^2 tiles take 5.96 ms, against 63.8 ms with separate column, separation
// and accumulation passes and FP64 sums for every tile.  The filters and den^2 are made once per
// PSF, not per tile.  Tiles are taken in chunks whose pairs fit the plan's pool;
// where not even one tile's do, the pairs are taken in groups and U is carried.

struct CArgs {
    const float* F;         // [n_frames]
    const float* sig;       // [n_frames]
    int n_frames;
    int j0;                 // first frame of the group
    int n_pairs;            // pairs of the group
    int first, last;        // whether the group is the first, the last of the frames
    int psf_tiles;          // tiles of the chunk, or 1 when every tile shares a frame's PSF
    int n_tiles;            // tiles of the chunk
    double eps2;
    float2* filt;           // [psf tile][pair][T kx][T ky] w_0 conj P_0 - i w_1 conj P_1
    double2* den;           // [psf tile][T / 2 + 1][T] (den^2, max |P|^2), carried between groups
    float2* dtab;           // [psf tile][T / 2 + 1][T] (den, den / F_R), 0 below the floor
    const float2* z;        // [pair][tile] blocked row transforms
    float2* zs;             // U carried between groups, then half-inverted S
    float2* zr;             // half-inverted R
    float2* zp;             // half-inverted P_R, or null
    const float2* tw;
};

// Frame j's matched-filter weights: F / s^2 for the score, F^2 / s^2 for den^2
// (a frame with s <= 0, or past the last frame, has none).
__host__ __device__ __forceinline__ void frame_weights(const float* F, const float* sig, int n, int j, float& w,
                                                       double& a) {
    w = 0.0f;
    a = 0.0;
    if (j < n && sig[j] > 0.0f) {
        w = F[j] / (sig[j] * sig[j]);
        a = (double)F[j] * F[j] / ((double)sig[j] * sig[j]);
    }
}

// The filter of a pair at k (MIRROR: at -k, where the transforms are conjugate) from
// w_0 P_0(k) and w_1 P_1(k).
template <bool MIRROR>
__host__ __device__ __forceinline__ float2 coadd_filter(float2 p0, float2 p1) {
    // conj(p0) - i conj(p1); with p -> conj p: p0 - i p1
    return MIRROR ? make_float2(p0.x + p1.y, p0.y - p1.x) : make_float2(p0.x - p1.y, -p0.y - p1.x);
}

__host__ __device__ __forceinline__ void coadd_den(double2 P, double a, double2& acc2) {
    const double q = P.x * P.x + P.y * P.y;
    acc2.x += a * q;
    if (a > 0.0 && q > acc2.y) acc2.y = q;
}

__host__ __device__ __forceinline__ float2 scaled(float w, double2 P) {
    const float2 p = f2(P);
    return make_float2(w * p.x, w * p.y);
}

// Accumulate one frame pair at frequency k: A = z1(k), B = z1(-k), C = z2(k),
// E = z2(-k), with z2 = DFT[P_0 + i P_1] (the CPU driver's form: the score is the
// conjugate-symmetric part of U).
[[maybe_unused]] __host__ __device__ __forceinline__ void coadd_accum_point(float2 A, float2 B, double2 C, double2 E, float w0,
                                                           float w1, double a0, double a1, float2& acc,
                                                           double2& acc2) {
    const double2 P0 = make_double2(0.5 * (C.x + E.x), 0.5 * (C.y - E.y));
    const double2 P1 = make_double2(0.5 * (C.y + E.y), -0.5 * (C.x - E.x));
    const float2 p0 = scaled(w0, P0), p1 = scaled(w1, P1);
    const float2 q = fft::cmul(coadd_filter<false>(p0, p1), A), m = fft::cmul(coadd_filter<true>(p0, p1), B);
    acc.x += 0.5f * (q.x + m.x);
    acc.y += 0.5f * (q.y - m.y);
    coadd_den(P0, a0, acc2);
    coadd_den(P1, a1, acc2);
}

// (den, den / F_R) at a frequency, 0 below the floor.
__host__ __device__ __forceinline__ float2 coadd_norm_point(double2 acc2, double FR, double eps2) {
    const double den = sqrt(acc2.x);
    return acc2.y >= eps2 && den > 0.0 ? make_float2((float)den, (float)(den / FR)) : make_float2(0.0f, 0.0f);
}

__host__ __device__ __forceinline__ float2 coadd_whiten(float2 Sh, float d) {
    return d > 0.0f ? make_float2(Sh.x / d, Sh.y / d) : make_float2(0.0f, 0.0f);
}

// The last step at frequency k: W = S + i R and the P_R spectrum (the CPU driver's form).
[[maybe_unused]] __host__ __device__ __forceinline__ void coadd_final_point(float2 Sh, double2 acc2, double FR, double eps2, float2& W,
                                                           float2& PRh) {
    const float2 d = coadd_norm_point(acc2, FR, eps2);
    const float2 Rh = coadd_whiten(Sh, d.x);
    PRh = make_float2(d.y, 0.0f);
    W = make_float2(Sh.x - Rh.y, Sh.y + Rh.x);
}

// Filters of the group's pairs and den^2.  Grid psf_tiles * ceil((T / 2 + 1) / PSEQ).
template <int T>
__global__ void __launch_bounds__(PSEQ * fft::Reg<T>::LANES) coadd_psf_cols_kernel(PsfArgs a, CArgs q) {
    using Rg = fft::Reg<T>;
    extern __shared__ __align__(16) unsigned char fft_smem[];
    double2* sm = reinterpret_cast<double2*>(fft_smem);
    constexpr int HW = T / 2 + 1, NB = (HW + PSEQ - 1) / PSEQ, L = Rg::LANES;
    const int c = threadIdx.x % PSEQ, lane = threadIdx.x / PSEQ;
    const long t = blockIdx.x / NB;
    const int kx = (int)(blockIdx.x - t * NB) * PSEQ + c;
    double2* b0 = sm + c;
    double2* b1 = sm + PSEQ * Rg::PT + c;
    const fft::TwTab<T> tw{a.tw, lane};
    const long h0 = (t * HW + kx) * T + lane;
    double2 acc[8], v[8];
#pragma unroll
    for (int m = 0; m < 8; m++)
        acc[m] = q.first || kx >= HW ? make_double2(0.0, 0.0) : q.den[h0 + m * L];
#pragma unroll 1
    for (int p = 0; p < q.n_pairs; p++) {
        float w0, w1;
        double a0, a1;
        frame_weights(q.F, q.sig, q.n_frames, q.j0 + 2 * p, w0, a0);
        frame_weights(q.F, q.sig, q.n_frames, q.j0 + 2 * p + 1, w1, a1);
        const double2* rows = a.rows + (t * a.n_pairs + p) * 2 * a.ps * HW;
        float2 p0[8];
        psf_column<T>(v, rows, a.ps, kx, tw, b0, b1, lane);
#pragma unroll
        for (int m = 0; m < 8; m++) {
            p0[m] = scaled(w0, v[m]);
            coadd_den(v[m], a0, acc[m]);
        }
        psf_column<T>(v, rows + (long)a.ps * HW, a.ps, kx, tw, b0, b1, lane);
        float2* f = q.filt + (t * q.n_pairs + p) * T * T;
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const int ky = lane + m * L;
            const float2 p1 = scaled(w1, v[m]);
            coadd_den(v[m], a1, acc[m]);
            if (kx < HW) f[(long)kx * T + ky] = coadd_filter<false>(p0[m], p1);
            if (kx > 0 && kx < T / 2) f[(long)(T - kx) * T + ((T - ky) & (T - 1))] = coadd_filter<true>(p0[m], p1);
        }
    }
    if (kx >= HW) return;
    double fr2 = 0.0;
    for (int j = 0; j < q.n_frames; j++) {
        float w;
        double aj;
        frame_weights(q.F, q.sig, q.n_frames, j, w, aj);
        fr2 += aj;
    }
    const double FR = sqrt(fr2);
#pragma unroll
    for (int m = 0; m < 8; m++) {
        if (q.last) q.dtab[h0 + m * L] = coadd_norm_point(acc[m], FR, q.eps2);
        else q.den[h0 + m * L] = acc[m];
    }
}

// Columns of the chunk's tiles over the group's pairs.  Grid n_tiles * T / CB.
template <int T>
__global__ void __launch_bounds__(fft::Reg<T>::THREADS, min_ctas<T>()) coadd_col_kernel(CArgs a) {
    using Rg = fft::Reg<T>;
    constexpr int CB = Rg::CB, L = Rg::LANES, NB = T / CB, HW = T / 2 + 1;
    extern __shared__ __align__(16) unsigned char fft_smem[];
    float2* sm = reinterpret_cast<float2*>(fft_smem);
    const int c = threadIdx.x % CB, lane = threadIdx.x / CB;
    const int t = blockIdx.x / NB, xb = blockIdx.x - t * NB, kx = xb * CB + c;
    const long blk = ((long)t * NB + xb) * T * CB + (long)lane * CB + c;
    const long pt = a.psf_tiles == 1 ? 0 : t;
    const float2* z = a.z + blk;
    const float2* f = a.filt + pt * a.n_pairs * T * T + (long)kx * T + lane;
    const fft::TwReg<T> tw(a.tw, lane);
    float2* b0 = sm + c;
    float2* b1 = sm + CB * Rg::PT + c;
    float2 u[8], v[8], nx[8];
#pragma unroll
    for (int m = 0; m < 8; m++) nx[m] = __ldcs(z + m * L * CB);
#pragma unroll
    for (int m = 0; m < 8; m++) u[m] = a.first ? make_float2(0.0f, 0.0f) : a.zs[blk + m * L * CB];
#pragma unroll 1
    for (int p = 0; p < a.n_pairs; p++) {
#pragma unroll
        for (int m = 0; m < 8; m++) v[m] = nx[m];
        float2 g[8];
#pragma unroll
        for (int m = 0; m < 8; m++) g[m] = __ldg(f + m * L);
        z += (long)a.n_tiles * T * T;
        f += T * T;
        if (p + 1 < a.n_pairs) {                           // the next pair's rows arrive during this one's transform
#pragma unroll
            for (int m = 0; m < 8; m++) nx[m] = __ldcs(z + m * L * CB);
        }
        fft::fft_reg<T, -1, CB>(v, tw, b0, b1, lane);
#pragma unroll
        for (int m = 0; m < 8; m++) {
            u[m].x += g[m].x * v[m].x - g[m].y * v[m].y;
            u[m].y += g[m].x * v[m].y + g[m].y * v[m].x;
        }
    }
    if (!a.last) {
#pragma unroll
        for (int m = 0; m < 8; m++) a.zs[blk + m * L * CB] = u[m];
        return;
    }
    const bool mir = kx > T / 2;
    const float2* d = a.dtab + (pt * HW + (mir ? T - kx : kx)) * T;
    float dr[8];
#pragma unroll
    for (int m = 0; m < 8; m++) {
        const int ky = lane + m * L;
        const float2 q = __ldg(d + (mir ? (T - ky) & (T - 1) : ky));
        v[m] = coadd_whiten(u[m], q.x);
        dr[m] = q.y;
    }
    fft::fft_reg<T, 1, CB>(u, tw, b0, b1, lane);
#pragma unroll
    for (int m = 0; m < 8; m++) a.zs[blk + m * L * CB] = u[m];
    fft::fft_reg<T, 1, CB>(v, tw, b0, b1, lane);
#pragma unroll
    for (int m = 0; m < 8; m++) a.zr[blk + m * L * CB] = v[m];
    if (a.zp) {
#pragma unroll
        for (int m = 0; m < 8; m++) v[m] = make_float2(dr[m], 0.0f);
        fft::fft_reg<T, 1, CB>(v, tw, b0, b1, lane);
#pragma unroll
        for (int m = 0; m < 8; m++) a.zp[blk + m * L * CB] = v[m];
    }
}

// sigma_S (sqrt(sum_j F_j^2 / s_j^2 sum P_tj^2), one CTA per PSF set) and F_R.  A
// thread sums a stamp's pixels tid, tid + 256, ...; a single thread per tile took
// 2.0 ms of a 30-frame coadd.
__global__ void __launch_bounds__(256) coadd_norm_kernel(const float* psfs, int ps, int psf_tiles, int n_tiles,
                                                         const float* F, const float* sig, int n_frames,
                                                         double* sigma_S, double* F_R) {
    __shared__ double red[8], all;
    const int pp = ps * ps;
    const float* pt = psfs + (long)blockIdx.x * n_frames * pp;
    double v = 0.0, fr2 = 0.0;
    for (int j = 0; j < n_frames; j++, pt += pp) {
        float w;
        double aj, s2 = 0.0;
        frame_weights(F, sig, n_frames, j, w, aj);
        for (int i = threadIdx.x; i < pp; i += 256) s2 += (double)pt[i] * pt[i];
        v += aj * s2;
        fr2 += aj;
    }
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < 8; i++) s += red[i];
        all = sqrt(s);
        if (F_R && blockIdx.x == 0) *F_R = sqrt(fr2);
    }
    __syncthreads();
    if (!sigma_S) return;
    if (psf_tiles > 1 || n_tiles == 1) {
        if (threadIdx.x == 0) sigma_S[blockIdx.x] = all;
    } else {
        for (int t = threadIdx.x; t < n_tiles; t += 256) sigma_S[t] = all;
    }
}

// How a coadd of n tiles and P frame pairs is cut to fit `avail` bytes: tiles per chunk
// and pairs per group (all of them, unless not even one tile's pairs fit).
struct CoaddCut {
    int tiles, group;
    size_t z, filt, rows, den, dtab;   // bytes: per (pair, tile); per (pair, PSF tile) x 2; per PSF tile x 2
    size_t out;                        // bytes per tile: half-inverted outputs
};
__host__ CoaddCut coadd_cut(int T, int n, int pairs, int ps, bool shared, bool pr, size_t avail) {
    CoaddCut c;
    const size_t px = (size_t)T * T, half = (size_t)(T / 2 + 1) * T;
    c.z = c.filt = 8 * px;
    c.rows = (size_t)2 * ps * (T / 2 + 1) * 16;
    c.den = 16 * half;
    c.dtab = 8 * half;
    c.out = (pr ? 24 : 16) * px;
    const size_t per_psf = c.den + c.dtab;                                  // + group * (filt + rows)
    const size_t fixed = shared ? per_psf + pairs * (c.filt + c.rows) : 0;
    const size_t tile = c.out + pairs * c.z + (shared ? 0 : per_psf + pairs * (c.filt + c.rows));
    const size_t fit = avail > fixed ? (avail - fixed) / tile : 0;
    if (fit >= 1) {
        const int chunks = (int)((n + fit - 1) / fit);
        c.tiles = (n + chunks - 1) / chunks;
        c.group = pairs;
    } else {
        c.tiles = 1;
        c.group = (int)((avail - per_psf - c.out) / (c.z + c.filt + c.rows));
    }
    return c;
}

struct CoaddCall {
    const float* stack;
    long frame_stride, pitch;
    int w, h;
    const int* origins;
    int n_tiles;
    const float* psfs;
    int ps;
    bool shared;
    float* S;
    float* R;
    float* PR;
    double* F_R;
    double* sigma_S;
};

template <int T>
int run_coadd(argus_proper_plan* p, const CoaddCall& c, CArgs a, cudaStream_t s) {
    using Rg = fft::Reg<T>;
    const int pairs = (a.n_frames + 1) / 2, pp = c.ps * c.ps;
    const CoaddCut cut = coadd_cut(T, c.n_tiles, pairs, c.ps, c.shared, c.PR != nullptr, pool_bytes(T, p->max_tiles));
    if (cut.group < 1) return ARGUS_ERR_UNSUPPORTED;       // cannot happen: the pool holds one pair of one tile
    const size_t npsf = c.shared ? 1 : cut.tiles;
    unsigned char* q = p->pool;
    double2* rowtmp = reinterpret_cast<double2*>(q); q += npsf * cut.group * cut.rows;
    a.den = reinterpret_cast<double2*>(q); q += npsf * cut.den;
    a.dtab = reinterpret_cast<float2*>(q); q += npsf * cut.dtab;
    a.filt = reinterpret_cast<float2*>(q); q += npsf * cut.group * cut.filt;
    float2* z = reinterpret_cast<float2*>(q); q += (size_t)cut.tiles * cut.group * cut.z;
    a.zs = reinterpret_cast<float2*>(q);
    a.zr = a.zs + (size_t)cut.tiles * T * T;
    a.zp = c.PR ? a.zr + (size_t)cut.tiles * T * T : nullptr;
    a.z = z;
    a.tw = p->tw32;
    for (int t0 = 0; t0 < c.n_tiles; t0 += cut.tiles) {
        a.n_tiles = c.n_tiles - t0 < cut.tiles ? c.n_tiles - t0 : cut.tiles;
        a.psf_tiles = c.shared ? 1 : a.n_tiles;
        const long o = (long)t0 * T * T;
        for (int g0 = 0; g0 < pairs; g0 += cut.group) {
            a.n_pairs = pairs - g0 < cut.group ? pairs - g0 : cut.group;
            a.j0 = 2 * g0;
            a.first = g0 == 0;
            a.last = g0 + a.n_pairs == pairs;
            const int second = (a.n_frames - a.j0) / 2 < a.n_pairs ? (a.n_frames - a.j0) / 2 : a.n_pairs;
            if (!c.shared || cut.group < pairs || t0 == 0) {          // shared filters serve every chunk
                PsfArgs f;
                f.tile_stride = c.shared ? 0 : (long)a.n_frames * pp;
                f.p0 = c.psfs + (c.shared ? 0 : (long)t0 * a.n_frames * pp) + (long)a.j0 * pp;
                f.p1 = f.p0 + pp;
                f.pair_stride = 2L * pp;
                f.n_second = second;
                f.n_pairs = a.n_pairs;
                f.ps = c.ps;
                f.tw = p->tw64;
                f.rows = rowtmp;
                const long rb = (long)a.psf_tiles * a.n_pairs * ((c.ps + PSEQ - 1) / PSEQ);
                psf_rows_kernel<T><<<(unsigned)rb, PSEQ * Rg::LANES, psf_smem<T>(), s>>>(f);
                coadd_psf_cols_kernel<T><<<(unsigned)a.psf_tiles * psf_col_blocks<T>(), PSEQ * Rg::LANES, psf_smem<T>(), s>>>(f, a);
                argus_count_launch(2);
            }
            RowArgs r;
            r.s0 = c.stack + a.j0 * c.frame_stride;
            r.s1 = r.s0 + c.frame_stride;
            r.pair_stride = 2 * c.frame_stride;
            r.n_second = second;
            r.pitch = c.pitch; r.w = c.w; r.h = c.h;
            r.org = c.origins + 2L * t0;
            r.org_stride = 2;
            r.n_tiles = a.n_tiles;
            r.tw = p->tw32;
            r.z = z;
            launch_rows<T>(r, a.n_pairs, s);
            coadd_col_kernel<T><<<(unsigned)a.n_tiles * (T / Rg::CB), Rg::THREADS, img_smem<T>(), s>>>(a);
            argus_count_launch(1);
        }
        launch_inv<T>(a.zs, a.zr, c.S + o, c.R + o, a.n_tiles, p->tw32, s);
        if (c.PR) launch_inv<T>(a.zp, nullptr, c.PR + o, nullptr, a.n_tiles, p->tw32, s);
    }
    coadd_norm_kernel<<<c.shared ? 1 : c.n_tiles, 256, 0, s>>>(c.psfs, c.ps, c.shared ? 1 : c.n_tiles, c.n_tiles, a.F,
                                                              a.sig, a.n_frames, c.sigma_S, c.F_R);
    argus_count_launch(1);
    return argus_launch_status();
}

template <typename K> bool dyn_smem(K* kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

template <int T>
bool set_smem() {
    const size_t i = img_smem<T>(), p = psf_smem<T>();
    return dyn_smem(row_fwd_kernel<T>, i) && dyn_smem(row_inv_kernel<T>, i) &&
           dyn_smem(row_inv_real_kernel<T, true>, i) && dyn_smem(row_inv_real_kernel<T, false>, i) && dyn_smem(zogy_col_kernel<T>, 2 * i) &&
           dyn_smem(coadd_col_kernel<T>, i) && dyn_smem(psf_rows_kernel<T>, p) && dyn_smem(zogy_psf_cols_kernel<T>, p) &&
           dyn_smem(coadd_psf_cols_kernel<T>, p);
}

}  // namespace

extern "C" int argus_proper_plan_create(int device, int tile, int max_tiles, argus_proper_plan** out) {
    if (!out || (tile != 256 && tile != 512 && tile != 1024) || max_tiles < 1 || max_tiles > 65536)
        return ARGUS_ERR_ARG;
    *out = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return ARGUS_ERR_CUDA;
    const bool smem_ok = tile == 256 ? set_smem<256>() : tile == 512 ? set_smem<512>() : set_smem<1024>();
    if (!smem_ok) return ARGUS_ERR_CUDA;
    argus_proper_plan* p = (argus_proper_plan*)calloc(1, sizeof(argus_proper_plan));
    if (!p) return ARGUS_ERR_NOMEM;
    p->device = device;
    p->tile = tile;
    p->max_tiles = max_tiles;
    const size_t parts = (size_t)max_tiles * (tile == 256 ? zogy_blocks<256>() : tile == 512 ? zogy_blocks<512>() : zogy_blocks<1024>());
    bool ok = cudaMalloc((void**)&p->pool, pool_bytes(tile, max_tiles)) == cudaSuccess;
    ok = ok && cudaMalloc((void**)&p->psd, parts * sizeof(double)) == cudaSuccess;
    ok = ok && cudaMalloc((void**)&p->tw32, (size_t)tile * sizeof(float2)) == cudaSuccess;
    ok = ok && cudaMalloc((void**)&p->tw64, (size_t)tile * sizeof(double2)) == cudaSuccess;
    if (ok) {
        // twiddles e^{-2 pi i m / T} in double on the host, rounded once to float
        double2* h64 = (double2*)malloc((size_t)tile * sizeof(double2));
        float2* h32 = (float2*)malloc((size_t)tile * sizeof(float2));
        ok = h64 && h32;
        if (ok) {
            const double two_pi = 6.283185307179586476925286766559;
            for (int m = 0; m < tile; m++) {
                const double ang = two_pi * (double)m / (double)tile;
                h64[m] = make_double2(std::cos(ang), -std::sin(ang));
                h32[m] = make_float2((float)h64[m].x, (float)h64[m].y);
            }
            ok = cudaMemcpy(p->tw64, h64, (size_t)tile * sizeof(double2), cudaMemcpyHostToDevice) == cudaSuccess &&
                 cudaMemcpy(p->tw32, h32, (size_t)tile * sizeof(float2), cudaMemcpyHostToDevice) == cudaSuccess;
        }
        free(h64);
        free(h32);
    }
    if (!ok) {
        cudaFree(p->pool); cudaFree(p->psd); cudaFree(p->tw32); cudaFree(p->tw64);
        free(p);
        return ARGUS_ERR_NOMEM;
    }
    *out = p;
    return ARGUS_OK;
}

extern "C" int argus_proper_plan_destroy(argus_proper_plan* p) {
    if (!p) return ARGUS_ERR_ARG;
    cudaSetDevice(p->device);
    cudaFree(p->pool); cudaFree(p->psd); cudaFree(p->tw32); cudaFree(p->tw64);
    free(p);
    return ARGUS_OK;
}

// May a call without PSFs reuse the transforms a plan holds?  held: the plan's psf_tiles
// (> 0 that many tiles' own pairs, -1 one shared pair, 0 none).  A per-tile call needs at
// least n_tiles per-tile pairs; a shared call needs the shared pair.
__host__ __device__ inline bool zogy_psf_reuse_ok(int held, int psf_per_tile, int n_tiles) {
    return psf_per_tile ? (held >= 1 && n_tiles <= held) : held == -1;
}

extern "C" int argus_zogy(argus_proper_plan* plan, const float* N, const float* R, argus_shape shape,
                          const argus_zogy_tile* tiles, int n_tiles, const float* psf_n, const float* psf_r,
                          int psf_size, int psf_per_tile, float eps, float* D, float* S, float* P_D,
                          double* sigma_S, argus_stream stream) {
    if (!plan || !N || !R || !tiles || !D || !S || n_tiles < 1 || n_tiles > plan->max_tiles) return ARGUS_ERR_ARG;
    if (!psf_n != !psf_r || (psf_per_tile != 0 && psf_per_tile != 1)) return ARGUS_ERR_ARG;
    // what the plan holds: psf_tiles > 0 tiles of their own, -1 one shared pair, 0 nothing
    if (!psf_n && !zogy_psf_reuse_ok(plan->psf_tiles, psf_per_tile, n_tiles)) return ARGUS_ERR_ARG;
    if (psf_size < 1 || (psf_size & 1) == 0 || psf_size > 63 || !(eps >= 0.0f)) return ARGUS_ERR_ARG;
    int st = argus_check_shape(shape, (size_t)-1);
    if (st) return st;
    if (cudaSetDevice(plan->device) != cudaSuccess) return ARGUS_ERR_CUDA;
    ZArgs a;
    a.tiles = tiles; a.n_tiles = n_tiles;
    a.psf_tiles = psf_per_tile ? n_tiles : 1;
    a.eps2 = (double)eps * (double)eps;
    // FP32 moduli (a few ulps off) decide the floor outside these bounds; floors too small
    // for FP32 are always decided in FP64
    a.hi2 = a.eps2 < 1e-30 ? 1e-30f : (float)(1.0001 * a.eps2);
    a.lo2 = a.eps2 < 1e-30 ? -1.0f : (float)(0.9999 * a.eps2);
    a.sigma_S = sigma_S;
    RowArgs r;
    r.s0 = N; r.s1 = R; r.pair_stride = 0; r.n_second = 1; r.pitch = shape.pitch; r.w = shape.w; r.h = shape.h;
    r.org = reinterpret_cast<const int*>(tiles); r.org_stride = (int)(sizeof(argus_zogy_tile) / sizeof(int));
    r.n_tiles = n_tiles;
    PsfArgs f;
    f.p0 = psf_n; f.p1 = psf_r; f.tile_stride = (long)psf_size * psf_size; f.pair_stride = 0; f.n_second = 1;
    f.n_pairs = 1; f.ps = psf_size;
    const PsfArgs* pf = psf_n ? &f : nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    int rc;
    switch (plan->tile) {
        case 256: rc = run<256>(plan, a, r, pf, D, S, P_D, s); break;
        case 512: rc = run<512>(plan, a, r, pf, D, S, P_D, s); break;
        default: rc = run<1024>(plan, a, r, pf, D, S, P_D, s); break;
    }
    if (psf_n) plan->psf_tiles = rc != ARGUS_OK ? 0 : (psf_per_tile ? n_tiles : -1);
    return rc;
}

extern "C" int argus_proper_coadd(argus_proper_plan* plan, const float* stack, int n_frames, argus_shape shape,
                                  const int* origins, int n_tiles, const float* F, const float* sigma,
                                  const float* psfs, int psf_size, int psf_per_tile, float eps, float* S,
                                  float* R, float* P_R,
                                  double* F_R, double* sigma_S, argus_stream stream) {
    if (!plan || !stack || !origins || !F || !sigma || !psfs || !S || !R || n_tiles < 1 ||
        n_tiles > plan->max_tiles || n_frames < 1 || n_frames > ARGUS_MAX_FRAMES)
        return ARGUS_ERR_ARG;
    if (psf_size < 1 || (psf_size & 1) == 0 || psf_size > 63 || !(eps >= 0.0f)) return ARGUS_ERR_ARG;
    if (psf_per_tile != 0 && psf_per_tile != 1) return ARGUS_ERR_ARG;
    int st = argus_check_shape(shape, (size_t)-1);
    if (st) return st;
    if (cudaSetDevice(plan->device) != cudaSuccess) return ARGUS_ERR_CUDA;
    CoaddCall c;
    c.stack = stack; c.frame_stride = (long)shape.h * shape.pitch; c.pitch = shape.pitch;
    c.w = shape.w; c.h = shape.h; c.origins = origins; c.n_tiles = n_tiles;
    c.psfs = psfs; c.ps = psf_size; c.shared = !psf_per_tile || n_tiles == 1;
    c.S = S; c.R = R; c.PR = P_R; c.F_R = F_R; c.sigma_S = sigma_S;
    CArgs a;
    a.F = F; a.sig = sigma; a.n_frames = n_frames; a.eps2 = (double)eps * (double)eps;
    plan->psf_tiles = 0;                                   // the pool is about to hold frames' transforms
    cudaStream_t s = (cudaStream_t)stream;
    switch (plan->tile) {
        case 256: return run_coadd<256>(plan, c, a, s);
        case 512: return run_coadd<512>(plan, c, a, s);
        default: return run_coadd<1024>(plan, c, a, s);
    }
}
