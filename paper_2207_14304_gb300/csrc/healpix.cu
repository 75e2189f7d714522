// Frame to HEALPix segment resampling (paper Sec. 3.3 "Image Segmentation";
// Table 2, GPU stage "Image segmentation and resampling to HEALPix grid").
//
// The segment's nested index gives its base face and face coordinates (X, Y);
// image pixel (column c, row r) is the HEALPix pixel (X 2^k + c, Y 2^k + r) at
// NSIDE_seg 2^k, whose centre (the ring / longitude formulas of the nested
// layout) is projected into the frame by the gnomonic WCS and the frame is
// interpolated there (bilinear, nested lerps, coverage as in the coadd).  The
// geometry is FP64 (a 9576-pixel frame needs positions to 1e-9 of the field);
// the output is FP32.  Exact path: one thread per pixel.  Patch path (k >= 6):
// a CTA per 64 x 64 patch, exact positions at 4 x 8 nodes and bicubics between
// them in the equatorial belt, in fixed point (see healpix_patch_kernel).
#include "argus_internal.cuh"

#include <cmath>

namespace {

struct HpArgs {
    const float* frame;
    const uint8_t* flags;
    long pitch;
    int w, h;
    const long long* segs;
    int n_seg;
    long long nside_seg;
    int k;
    double n[3], e[3], u[3];   // tangent-plane basis at the WCS centre
    double cr, sr, inv_scale, cx, cy;
    float* out;
    uint8_t* cov;
    long long xmax, ymax;      // the frame's last column and row as positions of the patch path
    bool split;                // halves that reach out of the belt are healpix_exact_kernel's
    double far;                // a half with every node's direction below this along n lies off the frame
};

__host__ __device__ __forceinline__ void hp_sincospi(double t, double* s, double* c) {
#ifdef __CUDA_ARCH__
    sincospi(t, s, c);
#else
    *s = std::sin(M_PI * t);
    *c = std::cos(M_PI * t);
#endif
}

// A segment: its image's first pixel in the face, and that pixel's ring.
struct HpSeg {
    long long nside, x, y, jr;
    int jp;                    // 2 pi / 8 units of the face's first pixel column
    bool ok;                   // a pixel of this NSIDE
};
__host__ __device__ __forceinline__ HpSeg hp_seg(const HpArgs& a, long long seg) {
    const long long N = a.nside_seg, face = seg / (N * N), ipf = seg - face * N * N;
    HpSeg g;
    g.nside = N << a.k;
    g.ok = seg >= 0 && face < 12;
    g.x = g.y = 0;
    for (int b = 0; (1LL << b) < N; b++) {
        g.x |= ((ipf >> (2 * b)) & 1LL) << b;
        g.y |= ((ipf >> (2 * b + 1)) & 1LL) << b;
    }
    g.x <<= a.k;
    g.y <<= a.k;
    g.jr = (face < 4 ? 2 : (face < 8 ? 3 : 4)) * g.nside - g.x - g.y - 1;
    g.jp = (int)(face < 4 ? 2 * face + 1 : (face < 8 ? 2 * (face - 4) : 2 * (face - 8) + 1));
    return g;
}

// z and sin(theta) of ring jr.
__host__ __device__ __forceinline__ double2 hp_ring(long long nside, long long jr) {
    if (jr >= nside && jr <= 3 * nside) {                // equatorial belt
        const double z = (double)(2 * nside - jr) * 2.0 / (3.0 * (double)nside);
        return make_double2(z, sqrt((1.0 - z) * (1.0 + z)));
    }
    const long long nr = jr < nside ? jr : 4 * nside - jr;
    const double cap = (double)nr * (double)nr / (3.0 * (double)nside * (double)nside);
    return make_double2(jr < nside ? 1.0 - cap : -1.0 + cap, sqrt(cap * (2.0 - cap)));
}

// Frame position of the centre of pixel (c, r) of a valid segment, `ring` its ring's
// values, and its direction along n.  false when that is behind the tangent plane.
__host__ __device__ __forceinline__ bool hp_on_ring(const HpArgs& a, const HpSeg& g, int c, int r, double2 ring, double& x,
                                                    double& y, double& d) {
    const long long jr = g.jr - c - r;
    const bool north = jr < g.nside, south = jr > 3 * g.nside;
    const long long nr = north ? jr : (south ? 4 * g.nside - jr : g.nside);
    const long long kshift = north || south ? 0 : (jr - g.nside) & 1;
    long long jp = (g.jp * nr + (g.x + c) - (g.y + r) + 1 + kshift) / 2;
    if (jp > 4 * nr) jp -= 4 * nr;
    if (jp < 1) jp += 4 * nr;
    // phi = (jp - (kshift + 1) / 2) (pi / 2) / nr
    double sp, cp;
    hp_sincospi(((double)jp - 0.5 * (double)(kshift + 1)) / (2.0 * (double)nr), &sp, &cp);
    const double v0 = ring.y * cp, v1 = ring.y * sp, v2 = ring.x;
    d = v0 * a.n[0] + v1 * a.n[1] + v2 * a.n[2];
    if (!(d > 0.0)) return false;
    const double xi = (v0 * a.e[0] + v1 * a.e[1] + v2 * a.e[2]) / d;
    const double eta = (v0 * a.u[0] + v1 * a.u[1] + v2 * a.u[2]) / d;
    x = a.cx + (a.cr * xi + a.sr * eta) * a.inv_scale;
    y = a.cy + (-a.sr * xi + a.cr * eta) * a.inv_scale;
    return true;
}

__host__ __device__ __forceinline__ bool hp_on_ring(const HpArgs& a, const HpSeg& g, int c, int r, double2 ring, double& x,
                                                    double& y) {
    double d;
    return hp_on_ring(a, g, c, r, ring, x, y, d);
}

// The same of any segment number; false for one that is no pixel of this NSIDE.
__host__ __device__ __forceinline__ bool hp_pixel_xy(const HpArgs& a, long long seg, int c, int r, double& x, double& y) {
    const HpSeg g = hp_seg(a, seg);
    return g.ok && hp_on_ring(a, g, c, r, hp_ring(g.nside, g.jr - c - r), x, y);
}

// Whether the w x h pixels from (c, r) on lie wholly in the equatorial belt (ring index in
// [N, 3N]): the ring index falls with c and with r, so the first and the last pixel tell.
__host__ __device__ __forceinline__ bool hp_in_belt(const HpSeg& g, int c, int r, int w, int h) {
    const long long first = g.jr - c - r;
    return g.ok && first <= 3 * g.nside && first - (w - 1) - (h - 1) >= g.nside;
}

// Nested-lerp bilinear value of the frame at (x, y); false when not covered
// (outside [0, w-1] x [0, h-1], or a neighbour with a nonzero weight flagged
// or not finite).
__host__ __device__ __forceinline__ bool hp_bilinear(const HpArgs& a, double x, double y, float& v) {
    if (!(x >= 0.0 && y >= 0.0 && x <= (double)(a.w - 1) && y <= (double)(a.h - 1))) return false;
    const int x0 = (int)floor(x), y0 = (int)floor(y);
    const double tx = x - x0, ty = y - y0;
    const bool ux = tx > 0.0, uy = ty > 0.0;
    double q[4] = {0.0, 0.0, 0.0, 0.0};
    const bool used[4] = {true, ux, uy, ux && uy};
    for (int i = 0; i < 4; i++) {
        if (!used[i]) continue;
        const long p = (long)(y0 + (i >> 1)) * a.pitch + x0 + (i & 1);
        const float f = a.frame[p];
        if (!isfinite(f) || (a.flags && a.flags[p])) return false;
        q[i] = f;
    }
    const double top = q[0] + tx * (q[1] - q[0]);
    const double bot = q[2] + tx * (q[3] - q[2]);
    v = (float)(top + ty * (bot - top));
    return true;
}

// Interpolation of positions.  Along a segment-image row or column in the
// equatorial belt the frame position is a smooth function of the column or row:
// on pieces of 64 pixels a cubic through the exact FP64 positions at 0, 21, 42,
// 63 of the piece reproduces it to a few 1e-8 pixel (a sixteenth of that on
// pieces of 32).  Newton form: d[0] = f0, d[1] = f[t0,t1], d[2] = f[t0,t1,t2],
// d[3] = f[t0..t3] (the row form hp_cubic_* and hp_row_in_belt is what the CPU
// checks run).
[[maybe_unused]] constexpr int HP_PIECE = 64;
__host__ __device__ __forceinline__ int hp_node(int j) { return j == 0 ? 0 : (j == 1 ? 21 : (j == 2 ? 42 : 63)); }

[[maybe_unused]] __host__ __device__ __forceinline__ void hp_cubic_coeffs(const double* f, double* d) {
    const double f01 = (f[1] - f[0]) / 21.0, f12 = (f[2] - f[1]) / 21.0, f23 = (f[3] - f[2]) / 21.0;
    const double f012 = (f12 - f01) / 42.0, f123 = (f23 - f12) / 42.0;
    d[0] = f[0];
    d[1] = f01;
    d[2] = f012;
    d[3] = (f123 - f012) / 63.0;
}

[[maybe_unused]] __host__ __device__ __forceinline__ double hp_cubic_eval(const double* d, double t) {
    return d[0] + t * (d[1] + (t - 21.0) * (d[2] + (t - 42.0) * d[3]));
}

// Whether a whole segment-image row lies in the equatorial belt (where the
// row interpolation is used): ring indices of its two end pixels in [N, 3N].
[[maybe_unused]] __host__ __device__ __forceinline__ bool hp_row_in_belt(const HpArgs& a, long long seg, int r) {
    const long long N = a.nside_seg;
    const long long face = seg / (N * N);
    if (seg < 0 || face >= 12) return false;
    const long long ipf = seg - face * N * N;
    long long X = 0, Y = 0;
    for (int b = 0; (1LL << b) < N; b++) {
        X |= ((ipf >> (2 * b)) & 1LL) << b;
        Y |= ((ipf >> (2 * b + 1)) & 1LL) << b;
    }
    const long long nside = N << a.k, m = 1LL << a.k;
    const long long jrll = face < 4 ? 2 : (face < 8 ? 3 : 4);
    const long long iy = (Y << a.k) + r;
    const long long jr0 = jrll * nside - (X << a.k) - iy - 1;         // column 0
    const long long jr1 = jr0 - (m - 1);                              // column m - 1
    return jr1 >= nside && jr0 <= 3 * nside;
}

// ---------------------------------------------------------------------------
// Patch path (k >= 6).  A CTA takes 64 x 64 pixels of a segment image as two
// halves of 64 x 32.  One warp computes the exact FP64 positions of the 32 nodes
// (columns 0, 21, 42, 63; rows 0, 10, 21, 31 of each half).  Per half, each column's
// positions along the rows are a cubic through its values at the four node rows,
// kept as forward differences in 64-bit fixed point (2^-44 pixel), so a pixel's
// position costs three 64-bit additions per coordinate and no FP64: this part does
// two FP64 operations per clock and SM, and evaluating two FP64 cubics and three
// FP64 lerps per pixel took 3.80 ms for the 170 segments of a 9576 x 6388 frame; this
// takes 0.525 ms (the FP64 pipe 46 % busy with nodes and columns, issue slots 61 %).
// The frame pixels under the half (a rectangle around its nodes) are staged in
// shared memory once, NaN where flagged or not finite: the image axes lie
// diagonally across the frame, and gathering neighbours from global memory
// touches about 27 lines per warp load.  The lerps run on unevaluated FP32 pairs
// (about 2^-44 relative, then one rounding).  Halves not wholly in the belt (unless
// `split` leaves them to healpix_exact_kernel), with a node behind the tangent plane or
// beyond HP_FAR pixels take the exact path per pixel; halves whose rectangle exceeds
// HP_CAP pixels gather from global memory.  Halves whose nodes all lie farther from the
// tangent point than any frame pixel and the patch allow for (HpArgs::far) are zero
// throughout: segments of the whole sky, most of them behind the plane or far off, cost the
// exact path otherwise (4 segments of 1024 x 1024: 307 to 442 us, 649 to 807 without).
constexpr int HP_PATCH = 64, HP_HALF = 32, HP_FRAC = 44, HP_CAP = 10240;
constexpr double HP_FAR = 500000.0;      // positions in fixed point stay below 2^19

__host__ __device__ __forceinline__ int hp_node_row(int j) { return j == 0 ? 0 : (j == 1 ? 10 : (j == 2 ? 21 : 31)); }

// The last position of a frame's axis, or the largest there is where the frame goes on past 2^19.
__host__ inline long long hp_last(int size) {
    return size - 1 < 1 << (63 - HP_FRAC) ? (long long)(size - 1) << HP_FRAC : 0x7fffffffffffffffll;
}

// Lagrange weights of the node columns 0, 21, 42, 63 at each column of a patch, times 2^HP_FRAC.
struct HpWeights { double w[HP_PATCH][4]; };
constexpr HpWeights hp_make_weights() {
    HpWeights t{};
    for (int c = 0; c < HP_PATCH; c++)
        for (int j = 0; j < 4; j++) {
            double num = (double)(1LL << HP_FRAC), den = 1.0;
            for (int i = 0; i < 4; i++)
                if (i != j) {
                    num *= (double)(c - 21 * i);
                    den *= (double)(21 * (j - i));
                }
            t.w[c][j] = num / den;
        }
    return t;
}
__device__ const HpWeights hp_weights = hp_make_weights();

// A column's coordinate at a node row from the node columns' (in units of 2^-HP_FRAC).
__host__ __device__ __forceinline__ double hp_column(const double* w, double n0, double n1, double n2, double n3) {
    return ((w[0] * n0 + w[1] * n1) + w[2] * n2) + w[3] * n3;
}

// Forward differences at row 0 (unit steps) of the cubic through v[] at the node
// rows 0, 10, 21, 31: from its divided differences c1, c2, c3,
// p(r) = v0 + c1 r + c2 r (r - 10) + c3 r (r - 10) (r - 21).
__host__ __device__ __forceinline__ void hp_differences(const double* v, long long* d) {
    const double f01 = (v[1] - v[0]) * (1.0 / 10.0), f12 = (v[2] - v[1]) * (1.0 / 11.0), f23 = (v[3] - v[2]) * (1.0 / 10.0);
    const double f012 = (f12 - f01) * (1.0 / 21.0), f123 = (f23 - f12) * (1.0 / 21.0);
    const double c3 = (f123 - f012) * (1.0 / 31.0);
    // r (r - 10) has differences -9, 2; r (r - 10) (r - 21) has 180, -56, 6
    d[0] = (long long)v[0];
    d[1] = (long long)(f01 - 9.0 * f012 + 180.0 * c3);
    d[2] = (long long)(2.0 * f012 - 56.0 * c3);
    d[3] = (long long)(6.0 * c3);
}

// The differences q rows on from those at row 0.
__host__ __device__ __forceinline__ void hp_advance(const long long* f, int q, long long* d) {
    const int q2 = q * (q - 1) / 2, q3 = q * (q - 1) * (q - 2) / 6;
    d[0] = f[0] + q * f[1] + q2 * f[2] + q3 * f[3];
    d[1] = f[1] + q * f[2] + q2 * f[3];
    d[2] = f[2] + q * f[3];
    d[3] = f[3];
}
__host__ __device__ __forceinline__ void hp_step(long long* d) {
    d[0] += d[1];
    d[1] += d[2];
    d[2] += d[3];
}

// a + t (b - a) with t = th + tl, a = ah + al, b = bh + bl as unevaluated pairs.
struct F2p { float h, l; };
__host__ __device__ __forceinline__ F2p hp_lerp(F2p a, F2p b, float th, float tl) {
    const float d = b.h - a.h, bb = d + a.h;               // d + e = b.h - a.h exactly
    const float e = (b.h - bb) - (a.h - (bb - d)) + (b.l - a.l);
    const float p = th * d, pl = fmaf(th, d, -p) + (th * e + tl * d);
    const float s = a.h + p, q = s - a.h;                  // s + r = a.h + p exactly
    const float r = (a.h - (s - q)) + (p - q) + (pl + a.l);
    return {s, r};
}

// The frame between the pixels q00 (x0, y0), q01 (x0 + 1, y0), q10, q11 at the fractions fx, fy
// (fixed point; 24 + 20 bits as a pair).
__host__ __device__ __forceinline__ float hp_fixed_bilinear(float q00, float q01, float q10, float q11, long long fx, long long fy) {
    const float xh = (float)(int)(fx >> 20) * 0x1p-24f, xl = (float)(int)(fx & 0xfffff) * 0x1p-44f;
    const float yh = (float)(int)(fy >> 20) * 0x1p-24f, yl = (float)(int)(fy & 0xfffff) * 0x1p-44f;
    const F2p top = hp_lerp({q00, 0.0f}, {q01, 0.0f}, xh, xl), bot = hp_lerp({q10, 0.0f}, {q11, 0.0f}, xh, xl);
    const F2p r = hp_lerp(top, bot, yh, yl);
    return r.h + r.l;
}

__device__ __forceinline__ float hp_nan() { return __int_as_float(0x7fffffff); }

// Frame pixel (x, y), NaN where flagged or not finite.
__device__ __forceinline__ float hp_fetch(const HpArgs& a, int x, int y) {
    const long p = (long)y * a.pitch + x;
    const float f = __ldg(a.frame + p);
    const unsigned fl = a.flags ? __ldg(a.flags + p) : 0u;
    return (fabsf(f) <= 3.402823466e38f) & (fl == 0u) ? f : hp_nan();
}

__global__ void __launch_bounds__(256, 4) healpix_patch_kernel(HpArgs a) {
    __shared__ double nd[2][4][4][2];                      // [half][node row][node column][x, y]
    __shared__ long long dif[2][HP_PATCH][4];              // [x, y][column] forward differences of a half
    __shared__ int box[2][4];                              // staged rectangle of a half: x0, y0, x1, y1
    __shared__ int okh[2];                                 // half: 1 interpolated, 0 exact, 2 not this kernel's, 3 off the frame
    extern __shared__ float hp_smem[];                     // staged frame pixels
    const int tid = threadIdx.x, lane = tid & 31, col = tid & 63, grp = tid >> 6;
    const int ppr = 1 << (a.k - 6);                        // patches per row
    const long s = blockIdx.x / (ppr * ppr);
    const int pq = (int)(blockIdx.x - s * ppr * ppr);
    const int c0 = (pq % ppr) * HP_PATCH, rp = (pq / ppr) * HP_PATCH;
    const long m = 1L << a.k;
    const long long seg = a.segs[s];
    float* out = a.out + s * m * m;
    uint8_t* cov = a.cov ? a.cov + s * m * m : nullptr;
    if (tid < 32) {
        const int hf = lane >> 4, jr = (lane >> 2) & 3, jc = lane & 3;
        double x = 0.0, y = 0.0;
        const int c = c0 + hp_node(jc), r = rp + hf * HP_HALF + hp_node_row(jr);
        const HpSeg g = hp_seg(a, seg);
        const bool belt = hp_in_belt(g, c0, rp + hf * HP_HALF, HP_PATCH, HP_HALF);
        double d = 1.0;
        const bool ok = belt && hp_on_ring(a, g, c, r, hp_ring(g.nside, g.jr - c - r), x, y, d) && fabs(x) < HP_FAR && fabs(y) < HP_FAR;
        nd[hf][jr][jc][0] = x;
        nd[hf][jr][jc][1] = y;
        const unsigned half = hf ? 0xffff0000u : 0x0000ffffu;
        const bool all = (__ballot_sync(0xffffffffu, ok) & half) == half;
        const bool off = (__ballot_sync(0xffffffffu, d < a.far) & half) == half;
        const int xi = ok ? (int)floor(x) : 0, yi = ok ? (int)floor(y) : 0;
        int bx0 = xi, bx1 = xi, by0 = yi, by1 = yi;
        for (int o = 8; o > 0; o >>= 1) {                  // over the half's 16 lanes
            bx0 = min(bx0, __shfl_xor_sync(0xffffffffu, bx0, o));
            bx1 = max(bx1, __shfl_xor_sync(0xffffffffu, bx1, o));
            by0 = min(by0, __shfl_xor_sync(0xffffffffu, by0, o));
            by1 = max(by1, __shfl_xor_sync(0xffffffffu, by1, o));
        }
        if ((lane & 15) == 0) {
            okh[hf] = off ? 3 : (all ? 1 : (a.split && !belt ? 2 : 0));
            box[hf][0] = max(bx0 - 1, 0);
            box[hf][1] = max(by0 - 1, 0);
            box[hf][2] = min(bx1 + 2, a.w - 1);
            box[hf][3] = min(by1 + 2, a.h - 1);
        }
    }
    __syncthreads();
    for (int hf = 0; hf < 2; hf++) {
        const int r0 = rp + hf * HP_HALF;
        if (okh[hf] == 2) continue;                        // (the same for the whole CTA)
        if (okh[hf] == 3) {
            for (int i = 0; i < HP_HALF / 4; i++) {
                const long e = (long)(r0 + grp * (HP_HALF / 4) + i) * m + c0 + col;
                out[e] = 0.0f;
                if (cov) cov[e] = 0;
            }
            continue;
        }
        if (!okh[hf]) {
            for (int i = 0; i < HP_HALF / 4; i++) {
                const int r = r0 + grp * (HP_HALF / 4) + i;
                double x, y;
                float v = 0.0f;
                const bool ok = hp_pixel_xy(a, seg, c0 + col, r, x, y) && hp_bilinear(a, x, y, v);
                const long e = (long)r * m + c0 + col;
                out[e] = ok ? v : 0.0f;
                if (cov) cov[e] = ok ? 1 : 0;
            }
            continue;
        }
        if (tid < 2 * HP_PATCH) {                          // grp 0: x, grp 1: y
            double v[4];
            for (int j = 0; j < 4; j++)
                v[j] = hp_column(hp_weights.w[col], nd[hf][j][0][grp], nd[hf][j][1][grp], nd[hf][j][2][grp], nd[hf][j][3][grp]);
            long long d[4];
            hp_differences(v, d);
            for (int i = 0; i < 4; i++) dif[grp][col][i] = d[i];
        }
        const int bx0 = box[hf][0], by0 = box[hf][1], bw = box[hf][2] - bx0 + 1, bh = box[hf][3] - by0 + 1;
        // shared row pitch: neighbouring columns step by (dx, dy); with a pitch of 0 mod 32 their bank
        // is x, with 1 mod 32 it is x + y -- take the one that moves
        const double dx = nd[hf][0][3][0] - nd[hf][0][0][0], dy = nd[hf][0][3][1] - nd[hf][0][0][1];
        const int P = ((bw + 31) & ~31) + (2.0 * fabs(dx) < fabs(dy) ? 1 : 0);
        const bool staged = bw > 0 && bh > 0 && (long)P * bh <= HP_CAP;
        if (staged) {
            // a warp takes eight rows at a time (the last repeated), all their loads in flight
            for (int y0 = (tid >> 5) * 8; y0 < bh; y0 += 64)
                for (int x = lane; x < bw; x += 32) {
                    float f[8];
#pragma unroll
                    for (int i = 0; i < 8; i++) f[i] = hp_fetch(a, bx0 + x, by0 + min(y0 + i, bh - 1));
#pragma unroll
                    for (int i = 0; i < 8; i++) hp_smem[min(y0 + i, bh - 1) * P + x] = f[i];
                }
        }
        __syncthreads();
        long long d[2][4];
        hp_advance(dif[0][col], grp * (HP_HALF / 4), d[0]);        // the group's first row
        hp_advance(dif[1][col], grp * (HP_HALF / 4), d[1]);
        const long long xmax = a.xmax, ymax = a.ymax;
        long e = (long)(r0 + grp * (HP_HALF / 4)) * m + c0 + col;
#pragma unroll 2
        for (int i = 0; i < HP_HALF / 4; i++, e += m) {
            const long long X = d[0][0], Y = d[1][0];
            hp_step(d[0]);
            hp_step(d[1]);
            float v = 0.0f;
            bool ok = X >= 0 && Y >= 0 && X <= xmax && Y <= ymax;
            if (ok) {
                const int x0 = (int)(X >> HP_FRAC), y0 = (int)(Y >> HP_FRAC);
                constexpr long long FM = (1LL << HP_FRAC) - 1;
                const long long fx = X & FM, fy = Y & FM;
                const int sx = fx ? 1 : 0, sy = fy ? 1 : 0;     // neighbours with a nonzero weight
                float q00, q01, q10, q11;
                const int lx = x0 - bx0, ly = y0 - by0;
                if (staged && lx >= 0 && ly >= 0 && lx + sx < bw && ly + sy < bh) {
                    const float* p = hp_smem + ly * P + lx;
                    q00 = p[0];
                    q01 = p[sx];
                    q10 = p[sy * P];
                    q11 = p[sy * P + sx];
                } else {
                    q00 = hp_fetch(a, x0, y0);
                    q01 = hp_fetch(a, x0 + sx, y0);
                    q10 = hp_fetch(a, x0, y0 + sy);
                    q11 = hp_fetch(a, x0 + sx, y0 + sy);
                }
                v = hp_fixed_bilinear(q00, q01, q10, q11, fx, fy);
                ok = q00 == q00 && q01 == q01 && q10 == q10 && q11 == q11;
                if (ok && !isfinite(v))                    // differences beyond FP32: lerps in FP64
                    hp_bilinear(a, (double)X * 0x1p-44, (double)Y * 0x1p-44, v);
            }
            out[e] = ok ? v : 0.0f;
            if (cov) cov[e] = ok ? 1 : 0;
        }
        __syncthreads();                                   // the staged pixels and differences are done with
    }
}

// Halves that reach out of the belt, per pixel on the exact path: a CTA takes HX_ROWS rows
// of up to HX_COLS columns, a warp a row.  A pixel's ring is that of its whole
// antidiagonal, so the CTA makes the rings' z and sin(theta) (a division and a square root
// each) once; FP64 bounds the rest.  A 9576 x 6388 frame at a declination of 60 degrees in segments
// of 512 x 512: 8.22 ms (in the patch kernel's exact branch 10.1, a warp per row without the
// rings' table 9.69); a 1500 x 1100 frame in segments of 128 x 128, too few patches for the
// SMs: 50 us (185 and 52).
constexpr int HX_ROWS = 8, HX_COLS = 512;

__global__ void __launch_bounds__(32 * HX_ROWS) healpix_exact_kernel(HpArgs a) {
    __shared__ double2 ring[HX_COLS + HX_ROWS - 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long m = 1L << a.k;
    const int W = (int)min(m, (long)HX_COLS), per_row = (int)(m / W);
    const long per_seg = m / HX_ROWS * per_row;
    for (long unit = blockIdx.x; unit < a.n_seg * per_seg; unit += gridDim.x) {
        const long s = unit / per_seg;
        const int q = (int)(unit - s * per_seg), c0 = q % per_row * W, r0 = q / per_row * HX_ROWS, rh = r0 & -HP_HALF;
        const HpSeg g = hp_seg(a, a.segs[s]);
        if (hp_in_belt(g, c0, rh, W, HP_HALF)) continue;   // the same for the whole CTA
        __syncthreads();                                   // the last unit's rings are done with
        if (g.ok)
            for (int e = threadIdx.x; e < W + HX_ROWS - 1; e += blockDim.x) ring[e] = hp_ring(g.nside, g.jr - c0 - r0 - e);
        __syncthreads();
        const int r = r0 + warp;
        const long row = (s * m + r) * m;
        for (int c = c0 + lane; c < c0 + W; c += 32) {
            if (hp_in_belt(g, c & -HP_PATCH, rh, HP_PATCH, HP_HALF)) continue;       // the patch kernel's
            double x, y;
            float v = 0.0f;
            const bool ok = g.ok && hp_on_ring(a, g, c, r, ring[c - c0 + warp], x, y) && hp_bilinear(a, x, y, v);
            a.out[row + c] = ok ? v : 0.0f;
            if (a.cov) a.cov[row + c] = ok ? 1 : 0;
        }
    }
}

__global__ void __launch_bounds__(256) healpix_resample_kernel(HpArgs a) {
    const long m = 1L << a.k;
    const long total = (long)a.n_seg * m * m;
    for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
        const long s = e / (m * m);
        const long q = e - s * m * m;
        const int r = (int)(q >> a.k), c = (int)(q & (m - 1));
        double x, y;
        float v = 0.0f;
        const bool ok = hp_pixel_xy(a, a.segs[s], c, r, x, y) && hp_bilinear(a, x, y, v);
        a.out[e] = ok ? v : 0.0f;
        if (a.cov) a.cov[e] = ok ? 1 : 0;
    }
}

// Host side of the argument set: the tangent-plane basis from the WCS.
__host__ inline void hp_fill_wcs(HpArgs& a, const argus_wcs& w) {
    const double ca = std::cos(w.alpha0), sa = std::sin(w.alpha0), cd = std::cos(w.delta0), sd = std::sin(w.delta0);
    a.n[0] = cd * ca; a.n[1] = cd * sa; a.n[2] = sd;
    a.e[0] = -sa; a.e[1] = ca; a.e[2] = 0.0;
    a.u[0] = -sd * ca; a.u[1] = -sd * sa; a.u[2] = cd;
    a.cr = std::cos(w.rot);
    a.sr = std::sin(w.rot);
    a.inv_scale = 1.0 / w.scale;
    a.cx = w.cx;
    a.cy = w.cy;
}

// The farthest frame pixel's angle from the tangent point: its farthest corner's.
__host__ inline double hp_frame_radius(const HpArgs& a) {
    const double dx = std::fmax(std::fabs(a.cx), std::fabs(a.w - 1 - a.cx)), dy = std::fmax(std::fabs(a.cy), std::fabs(a.h - 1 - a.cy));
    return std::atan(std::hypot(dx, dy) / a.inv_scale);
}

// Whether every pixel of the frame lies in the equatorial belt, |sin(dec)| <= 2/3.
__host__ inline bool hp_frame_in_belt(const HpArgs& a) {
    return std::asin(std::fabs(a.n[2])) + hp_frame_radius(a) < std::asin(2.0 / 3.0);
}

// Where the directions begin that are off the frame with a whole half patch around them: a pixel
// of a half lies at most 11 columns and 5 rows from a node, steps of at most 1.07 / NSIDE each
// in the belt.
__host__ inline double hp_far(const HpArgs& a) {
    return std::cos(std::fmin(hp_frame_radius(a) + 32.0 / ((double)a.nside_seg * (1 << a.k)), M_PI));
}

}  // namespace

extern "C" int argus_healpix_resample(const float* frame, const uint8_t* flags, argus_shape shape, argus_wcs wcs,
                                      int nside_seg, int k, const long long* segs, int n_seg, float* out,
                                      uint8_t* coverage, argus_stream stream) {
    if (!frame || !segs || !out || n_seg < 1 || k < 0 || k > 12 || nside_seg < 1 || nside_seg > (1 << 17) ||
        (nside_seg & (nside_seg - 1)) || !(wcs.scale > 0.0))
        return ARGUS_ERR_ARG;
    if ((long long)nside_seg << k > (1LL << 29)) return ARGUS_ERR_ARG;
    int st = argus_check_shape(shape, (size_t)-1);
    if (st) return st;
    HpArgs a;
    a.frame = frame; a.flags = flags; a.pitch = shape.pitch; a.w = shape.w; a.h = shape.h;
    a.segs = segs; a.n_seg = n_seg; a.nside_seg = nside_seg; a.k = k; a.out = out; a.cov = coverage;
    a.xmax = hp_last(shape.w); a.ymax = hp_last(shape.h);
    hp_fill_wcs(a, wcs);
    if (k >= 6) {                                  // whole 64 x 64 patches
        const long long patches = (long long)n_seg << (2 * (k - 6));
        if (patches > 0x7fffffffLL) return ARGUS_ERR_ARG;
        const size_t smem = HP_CAP * sizeof(float);
        // a frame inside the belt has next to no pixel of a half that reaches out of it: one kernel takes
        // them all (a second launch would add 3 us or so to calls of 31); any other frame's halves go to a
        // kernel of their own (at declinations 45 to 80 1.2 to 3.7 times as fast)
        a.split = !hp_frame_in_belt(a);
        a.far = hp_far(a);
        healpix_patch_kernel<<<(unsigned)patches, 256, smem, (cudaStream_t)stream>>>(a);
        if (a.split) {
            const long m = 1L << k, units = (long)n_seg * (m / HX_ROWS) * (m < HX_COLS ? 1 : m / HX_COLS);
            healpix_exact_kernel<<<(unsigned)(units < 152L * 32 ? units : 152L * 32), 32 * HX_ROWS, 0, (cudaStream_t)stream>>>(a);
            argus_count_launch(1);
        }
    } else {
        const long total = (long)n_seg << (2 * k);
        long blocks = (total + 255) / 256;
        if (blocks > 152L * 32) blocks = 152L * 32;
        healpix_resample_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(a);
    }
    argus_count_launch(1);
    return argus_launch_status();
}
