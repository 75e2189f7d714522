// Median-filtered background map (paper Table 2, GPU timing "Median-filtered
// background map"; background maps held with the calibration frames, Sec. 3.2).
//
//   1. box_median_kernel: one CTA per box x box mesh box; the valid pixels
//      (flag 0, finite) stay in registers as order-preserving 32-bit keys and a
//      bracket around the middle key(s) is narrowed by counting; the box value is
//      their mean in FP64 (exact), or NaN when fewer than min_frac of the box's
//      pixels are valid.
//   2. mesh_filter_kernel: one thread per box; the median of the values that
//      exist in its filt x filt neighbourhood (clipped at the mesh edges), and the
//      mesh in FP32 for the map.
//   3. mesh_fill_kernel: one CTA; if some neighbourhood had no value, the median
//      of all box values goes there, by radix select on 64-bit keys of the
//      doubles, reading the mesh from global memory.
//   4. interp_kernel: the map, bilinear between box centres (mean pixel
//      coordinate of each box), constant beyond the outermost ones, in FP32,
//      four pixels per thread.
#include "argus_internal.cuh"

#include <cstring>

namespace {

constexpr int BM_THREADS = 256;
constexpr int BM_MAX_PER = 16;          // box <= 64: at most 16 pixels per thread
constexpr int FILL_THREADS = 1024;

struct BgArgs {
    const float* img;
    const uint8_t* flags;
    double* raw;        // [ny][nx] box medians (NaN: no value)
    double* mesh;       // [ny][nx] filtered
    float* meshf;       // [ny][nx] the filtered mesh rounded to FP32
    int* missing;       // [1] neighbourhoods without a value
    double* fill;       // [1] what they take, when there are any
    float* map;
    long pitch;
    int w, h, box, filt, nx, ny;
    float min_frac;
};

// Bit patterns on host and device (the host side serves the CPU checks).
__host__ __device__ __forceinline__ unsigned f32_bits(float v) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(v);
#else
    unsigned u;
    memcpy(&u, &v, 4);
    return u;
#endif
}
__host__ __device__ __forceinline__ float bits_f32(unsigned u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float v;
    memcpy(&v, &u, 4);
    return v;
#endif
}
__host__ __device__ __forceinline__ unsigned long long f64_bits(double v) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(v);
#else
    unsigned long long u;
    memcpy(&u, &v, 8);
    return u;
#endif
}
__host__ __device__ __forceinline__ double bits_f64(unsigned long long u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double v;
    memcpy(&v, &u, 8);
    return v;
#endif
}

// Order-preserving keys: a < b (as numbers, -0 before +0) iff key(a) < key(b).
__host__ __device__ __forceinline__ unsigned key32(float v) {
    const unsigned u = f32_bits(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__host__ __device__ __forceinline__ float unkey32(unsigned k) {
    return bits_f32((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
__host__ __device__ __forceinline__ unsigned long long key64(double v) {
    const unsigned long long u = f64_bits(v);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__host__ __device__ __forceinline__ double unkey64(unsigned long long k) {
    return bits_f64((k >> 63) ? (k & 0x7fffffffffffffffull) : ~k);
}

// The radix form of a box's selection, one thread of 256 at a time: what the CPU
// checks run (box_load, box_hist, box_le_min).
// One thread's share of a box: pixels tid, tid + 256, ... of the box as keys
// (ok = valid); returns the count of valid pixels.
[[maybe_unused]] __host__ __device__ __forceinline__ int box_load(const BgArgs& a, int bx, int by, int tid, unsigned* key, bool* ok) {
    const int x0 = bx * a.box, y0 = by * a.box;
    const int bw = min(a.box, a.w - x0), bh = min(a.box, a.h - y0);
    const int npx = bw * bh;
    int nv = 0;
#pragma unroll
    for (int j = 0; j < BM_MAX_PER; j++) {
        const int i = tid + j * BM_THREADS;
        ok[j] = false;
        key[j] = 0;
        if (i < npx) {
            const int yy = i / bw, xx = i - yy * bw;
            const long p = (long)(y0 + yy) * a.pitch + x0 + xx;
            const float v = a.img[p];
            if (isfinite(v) && (!a.flags || a.flags[p] == 0)) {
                ok[j] = true;
                key[j] = key32(v);
                nv++;
            }
        }
    }
    return nv;
}

// One thread's histogram contribution of a radix pass: add(bin) for each of its
// keys that matches the prefix decided so far.
template <typename Add>
[[maybe_unused]] __host__ __device__ __forceinline__ void box_hist(const unsigned* key, const bool* ok, unsigned mask, unsigned prefix,
                                                  int shift, Add add) {
#pragma unroll
    for (int j = 0; j < BM_MAX_PER; j++)
        if (ok[j] && (key[j] & mask) == prefix) add((int)((key[j] >> shift) & 255u));
}

// One thread's count of keys <= k1 and its smallest key above k1.
[[maybe_unused]] __host__ __device__ __forceinline__ void box_le_min(const unsigned* key, const bool* ok, unsigned k1, int& le,
                                                    unsigned& m) {
    le = 0;
    m = 0xffffffffu;
#pragma unroll
    for (int j = 0; j < BM_MAX_PER; j++) {
        if (!ok[j]) continue;
        if (key[j] <= k1) le++;
        else m = min(m, key[j]);
    }
}

// The median from the middle keys: n odd -> k1 == k2.
__host__ __device__ __forceinline__ double median_of_keys(unsigned k1, unsigned k2) {
    return 0.5 * ((double)unkey32(k1) + (double)unkey32(k2));
}

// Whether a box with n valid pixels of npx has a value.
__host__ __device__ __forceinline__ bool box_has_value(int n, int npx, float min_frac) {
    return n > 0 && (float)n >= min_frac * (float)npx;
}

// Block-wide sum of an int (every thread receives it); `red` holds 32 ints.
__device__ __forceinline__ int block_sum(int v, int* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = __reduce_add_sync(0xffffffffu, v);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    int t = 0;
    for (int i = 0; i < nw; i++) t += red[i];
    return t;
}

// Bin of the 256-bin histogram holding the k-th element (0-based) in bin
// order; k is reduced to the rank inside that bin.  Called by every thread,
// result broadcast through shared memory.
__device__ __forceinline__ int pick_bin(const int* hist, int& k, int* sh) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int c[8], s = 0;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            c[i] = hist[lane * 8 + i];
            s += c[i];
        }
        int incl = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        int run = incl - s;                      // elements in the bins before this lane's 8
        if (k >= run && k < incl) {              // exactly one lane
            int b = lane * 8;
            for (int i = 0; i < 8; i++, b++) {
                if (k < run + c[i]) break;
                run += c[i];
            }
            sh[0] = b;
            sh[1] = k - run;
        }
    }
    __syncthreads();
    const int b = sh[0];
    k = sh[1];
    __syncthreads();
    return b;
}

// Box medians, one CTA of 128 threads per box, NPL keys per thread (pixel e = tid +
// 128 j of the box; 0xffffffff, above every valid key, where there is none or it is
// invalid).  The middle keys are bracketed: (lo, hi] holds the ranks clo .. chi - 1,
// among them r1 = (n - 1) / 2 and r2 = n / 2.  A pass counts the keys up to two
// thresholds -- first two order statistics of 32 of the keys, then an interpolated
// guess with a margin of a few keys either side -- until at most 32 keys are left,
// which one warp sorts.  Four or five passes of two compares and adds per key and one
// barrier: 196 us on a 9576 x 6388 frame of 64-pixel boxes (issue slots 69 % busy), against
// 514 us for an 8-bit radix select, whose first pass is atomics to the few bins that a
// box's exponents fall in.  After CAREFUL passes the thresholds halve the bracket
// instead, so every box ends.  One warp per box with all 4096 keys in its registers
// needed 200 of them and waited on its loads eight warps to an SM.
constexpr int BOX_THREADS = 128, BOX_WARPS = BOX_THREADS / 32, CAREFUL = 10;

// The bracket and its next thresholds, the same for every thread; host-callable, so a CPU
// driver can run the same selection.
constexpr unsigned BOX_NONE = 0xffffffffu;                 // above every valid key
struct BoxBracket {
    unsigned lo, hi;         // the ranks r1, r2 lie in (lo, hi], or at the cut
    int clo, chi, r1, r2;    // ranks clo .. chi - 1 are in it
    unsigned t, u;           // thresholds of the next pass, t <= u
    bool split;              // r1 is the last key <= cut, r2 the first above
    unsigned cut;
    // of n valid keys; s0 <= s1 the first thresholds
    __host__ __device__ __forceinline__ void init(int n, unsigned s0, unsigned s1) {
        r1 = (n - 1) / 2;
        r2 = n / 2;
        lo = 0u;             // no valid key is 0 or above hi
        hi = BOX_NONE - 1u;
        clo = 0;
        chi = n;
        t = s0;
        u = s1;
        split = false;
        cut = 0u;
    }
    __host__ __device__ __forceinline__ bool useful() const { return t > lo && t < hi && u > lo && u < hi; }
    // the counts of keys <= t and <= u
    __host__ __device__ __forceinline__ void narrow(int ct, int cu) {
        if (ct <= r1) { lo = t; clo = ct; }
        else if (ct > r2) { hi = t; chi = ct; }
        else { split = true; cut = t; }
        if (cu <= r1) { if (u > lo) { lo = u; clo = cu; } }
        else if (cu > r2) { if (u < hi) { hi = u; chi = cu; } }
        else { split = true; cut = u; }
    }
    __host__ __device__ __forceinline__ bool done() const { return split || chi - clo <= 32 || hi - lo == 1u; }
    // thresholds after pass it
    __host__ __device__ __forceinline__ void next(int it) {
        const unsigned span = hi - lo;
        if (it >= CAREFUL) {
            t = u = lo + span / 2;
        } else {
            const float c = (float)(chi - clo), per = (float)span / c;
            const float g = ((float)(r1 - clo) + 0.75f) * per, m = fmaxf(8.0f, 1.5f * sqrtf(c)) * per;
            // (2^32 as a float at most: one below it at the most where the cast is asked for)
            const float top = fminf((float)(span - 1u), 4294967040.0f);
            t = lo + umin_(umax_(1u, (unsigned)fminf(fmaxf(g - m, 1.0f), top)), span - 1u);
            u = lo + umin_(umax_(1u, (unsigned)fminf(g + m, top)), span - 1u);
        }
    }
    // whether a key is left in the bracket
    __host__ __device__ __forceinline__ bool holds(unsigned key) const { return key - lo - 1u < hi - lo; }
    static __host__ __device__ __forceinline__ unsigned umin_(unsigned a, unsigned b) { return a < b ? a : b; }
    static __host__ __device__ __forceinline__ unsigned umax_(unsigned a, unsigned b) { return a > b ? a : b; }
};

// The lanes' values in ascending order over the lanes (bitonic).
__device__ __forceinline__ unsigned warp_sort(unsigned v, int lane) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const unsigned o = __shfl_xor_sync(0xffffffffu, v, j);
            const bool low = ((lane & j) == 0) == ((lane & k) == 0);
            v = low ? min(v, o) : max(v, o);
        }
    return v;
}

// Sums of c and d over the CTA; `part` alternates between two slots, so one barrier does.
__device__ __forceinline__ int2 box_sum2(int c, int d, int2 (*part)[BOX_WARPS], int& slot) {
    c = __reduce_add_sync(0xffffffffu, c);
    d = __reduce_add_sync(0xffffffffu, d);
    if ((threadIdx.x & 31) == 0) part[slot][threadIdx.x >> 5] = make_int2(c, d);
    __syncthreads();
    int2 s = make_int2(0, 0);
#pragma unroll
    for (int i = 0; i < BOX_WARPS; i++) {
        s.x += part[slot][i].x;
        s.y += part[slot][i].y;
    }
    slot ^= 1;
    return s;
}

template <int NPL>
__global__ void __launch_bounds__(BOX_THREADS) box_median_kernel(BgArgs a) {
    __shared__ int2 part[2][BOX_WARPS];
    __shared__ unsigned smp[2], cand[32], kk[2][BOX_WARPS];
    __shared__ int at;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x;
    const int by = b / a.nx, bx = b - by * a.nx;
    const int bw = min(a.box, a.w - bx * a.box), bh = min(a.box, a.h - by * a.box), npx = bw * bh;
    unsigned key[NPL];
    int nv = 0, slot = 0;
    {
        const int dq = BOX_THREADS / bw, dr = BOX_THREADS - dq * bw;   // pixel e + 128: dq rows and dr columns on
        int yy = tid / bw, xx = tid - yy * bw;
        const long base = (long)by * a.box * a.pitch + bx * a.box;
        constexpr int LB = NPL < 8 ? NPL : NPL % 8 ? 6 : 8;            // loads in flight per thread and image
        static_assert(NPL % LB == 0, "whole batches");
#pragma unroll
        for (int j0 = 0; j0 < NPL; j0 += LB) {
            float v[LB];
            unsigned f[LB];
#pragma unroll
            for (int j = 0; j < LB; j++) {
                const bool in = tid + BOX_THREADS * (j0 + j) < npx;
                const long p = base + (long)yy * a.pitch + xx;
                v[j] = in ? __ldg(a.img + p) : __int_as_float(0x7fffffff);
                f[j] = in && a.flags ? __ldg(a.flags + p) : 0u;
                yy += dq;
                xx += dr;
                if (xx >= bw) { xx -= bw; yy++; }
            }
#pragma unroll
            for (int j = 0; j < LB; j++) {
                const bool ok = (f[j] == 0u) & (fabsf(v[j]) <= 3.402823466e38f);     // finite
                key[j0 + j] = ok ? key32(v[j]) : BOX_NONE;
                nv += ok ? 1 : 0;
            }
        }
    }
    if (warp == 0) {
        const unsigned v = warp_sort(key[0], lane);
        if (lane == 9) smp[0] = v;
        if (lane == 22) smp[1] = v;
        if (lane == 0) at = 0;
    }
    const int n = box_sum2(nv, 0, part, slot).x;
    if (!box_has_value(n, npx, a.min_frac)) {
        if (tid == 0) a.raw[b] = __longlong_as_double(0x7ff8000000000000ll);     // NaN: no value
        return;
    }
    BoxBracket q;
    q.init(n, smp[0], smp[1]);
    for (int it = 0;; it++) {                              // the same for every thread
        if (q.useful()) {
            int c = 0, d = 0;
#pragma unroll
            for (int j = 0; j < NPL; j++) {
                c += key[j] <= q.t ? 1 : 0;
                d += key[j] <= q.u ? 1 : 0;
            }
            const int2 s = box_sum2(c, d, part, slot);
            q.narrow(s.x, s.y);
        }
        if (q.done()) break;
        q.next(it);
    }
    if (q.split) {
        unsigned m1 = 0u, m2 = BOX_NONE;
#pragma unroll
        for (int j = 0; j < NPL; j++) {
            if (key[j] <= q.cut) m1 = max(m1, key[j]);
            else m2 = min(m2, key[j]);
        }
        m1 = __reduce_max_sync(0xffffffffu, m1);
        m2 = __reduce_min_sync(0xffffffffu, m2);
        if (lane == 0) {
            kk[0][warp] = m1;
            kk[1][warp] = m2;
        }
        __syncthreads();
        if (tid == 0) {
            for (int i = 1; i < BOX_WARPS; i++) {
                m1 = max(m1, kk[0][i]);
                m2 = min(m2, kk[1][i]);
            }
            a.raw[b] = median_of_keys(m1, m2);
        }
    } else if (q.hi - q.lo == 1u) {
        if (tid == 0) a.raw[b] = median_of_keys(q.hi, q.hi);   // every key left is hi
    } else {
#pragma unroll
        for (int j = 0; j < NPL; j++)
            if (q.holds(key[j])) cand[atomicAdd(&at, 1)] = key[j];     // at most 32
        __syncthreads();
        if (warp == 0) {
            const unsigned v = warp_sort(lane < at ? cand[lane] : BOX_NONE, lane);
            const unsigned k1 = __shfl_sync(0xffffffffu, v, q.r1 - q.clo), k2 = __shfl_sync(0xffffffffu, v, q.r2 - q.clo);
            if (lane == 0) a.raw[b] = median_of_keys(k1, k2);
        }
    }
}

// The cells whose neighbourhood had no value (NaN in the mesh) take the median of
// the non-NaN box values by radix select over global memory (one CTA), 0 if there
// are none.  Leaves at once where there is no such cell, as in nearly every frame
// (the selection takes 90 us on 15,000 boxes).
__global__ void __launch_bounds__(FILL_THREADS) mesh_fill_kernel(BgArgs a) {
    __shared__ int hist[256];
    __shared__ int red[32];
    __shared__ int sh[2];
    __shared__ unsigned long long umin[32];
    if (*a.missing == 0) return;
    const int ncell = a.nx * a.ny;
    const auto fill_in = [&](double v) {
        if (threadIdx.x == 0) *a.fill = v;
        for (int i = threadIdx.x; i < ncell; i += FILL_THREADS)
            if (isnan(a.mesh[i])) {
                a.mesh[i] = v;
                a.meshf[i] = (float)v;
            }
    };
    int nv = 0;
    for (int i = threadIdx.x; i < ncell; i += FILL_THREADS) nv += isnan(a.raw[i]) ? 0 : 1;
    const int n = block_sum(nv, red);
    if (n == 0) {
        fill_in(0.0);
        return;
    }
    int k = (n - 1) / 2;
    unsigned long long prefix = 0, mask = 0;
    for (int shift = 56; shift >= 0; shift -= 8) {
        for (int i = threadIdx.x; i < 256; i += FILL_THREADS) hist[i] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < ncell; i += FILL_THREADS) {
            const double v = a.raw[i];
            if (isnan(v)) continue;
            const unsigned long long kk = key64(v);
            if ((kk & mask) == prefix) atomicAdd(&hist[(kk >> shift) & 255ull], 1);
        }
        __syncthreads();
        const int b = pick_bin(hist, k, sh);
        prefix |= (unsigned long long)b << shift;
        mask |= 255ull << shift;
    }
    const unsigned long long k1 = prefix;
    unsigned long long k2 = k1;
    if ((n & 1) == 0) {
        int le = 0;
        unsigned long long m = ~0ull;
        for (int i = threadIdx.x; i < ncell; i += FILL_THREADS) {
            const double v = a.raw[i];
            if (isnan(v)) continue;
            const unsigned long long kk = key64(v);
            if (kk <= k1) le++;
            else m = kk < m ? kk : m;
        }
        const int nle = block_sum(le, red);
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long t = __shfl_xor_sync(0xffffffffu, m, o);
            m = t < m ? t : m;
        }
        if ((threadIdx.x & 31) == 0) umin[threadIdx.x >> 5] = m;
        __syncthreads();
        unsigned long long mm = ~0ull;
        for (int i = 0; i < FILL_THREADS / 32; i++) mm = umin[i] < mm ? umin[i] : mm;
        k2 = nle >= n / 2 + 1 ? k1 : mm;
    }
    fill_in(0.5 * (unkey64(k1) + unkey64(k2)));
}

// The filtered value of box (cx, cy): the median of the values that exist in its
// filt x filt neighbourhood, else `fill`.
__host__ __device__ __forceinline__ double filter_cell(const double* raw, int nx, int ny, int cx, int cy, int filt,
                                                       double fill) {
    const int r = filt / 2;
    double v[49];
    int n = 0;
    for (int y = max(0, cy - r); y <= min(ny - 1, cy + r); y++) {
        for (int x = max(0, cx - r); x <= min(nx - 1, cx + r); x++) {
            const double t = raw[(long)y * nx + x];
            if (isnan(t)) continue;
            int i = n++;                           // insertion into the sorted prefix
            while (i > 0 && v[i - 1] > t) {
                v[i] = v[i - 1];
                i--;
            }
            v[i] = t;
        }
    }
    return n ? 0.5 * (v[(n - 1) / 2] + v[n / 2]) : fill;
}

__global__ void __launch_bounds__(256) mesh_filter_kernel(BgArgs a) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= a.nx * a.ny) return;
    const int cy = c / a.nx, cx = c - cy * a.nx;
    const double v = filter_cell(a.raw, a.nx, a.ny, cx, cy, a.filt, __longlong_as_double(0x7ff8000000000000ll));
    a.mesh[c] = v;
    a.meshf[c] = (float)v;
    if (isnan(v)) atomicAdd(a.missing, 1);
}

// Interpolation coordinate along one axis: lower box index i (upper i + 1) and
// weight t of the upper one, clamped beyond the outermost centres.
__host__ __device__ __forceinline__ void axis_weight(int p, int n, int box, int nb, int& i, float& t) {
    if (nb == 1) {
        i = 0;
        t = 0.0f;
        return;
    }
    // box i's centre is i box + (box - 1) / 2 (a half-integer for even boxes):
    // i = floor((2 p - (box - 1)) / (2 box)), exact in integers
    const int num = 2 * p - (box - 1);
    i = num >= 0 ? num / (2 * box) : 0;
    i = min(i, nb - 2);
    const float c0 = i * box + 0.5f * (float)(box - 1);
    const int e1 = min((i + 2) * box, n);
    const float c1 = 0.5f * (float)((i + 1) * box + e1 - 1);
    t = fminf(fmaxf(((float)p - c0) / (c1 - c0), 0.0f), 1.0f);
}

// Bilinear value from the mesh row r0 (lower box ix, next box ix + jx, next row
// + jy) in FP32 (what the CPU checks run; interp_kernel does the same per row).
[[maybe_unused]] __host__ __device__ __forceinline__ float bilinear(const double* r0, int ix, int jx, int jy, float tx, float ty) {
    const float m00 = (float)r0[ix], m01 = (float)r0[ix + jx];
    const float m10 = (float)r0[jy + ix], m11 = (float)r0[jy + ix + jx];
    const float top = m00 + (m01 - m00) * tx;
    const float bot = m10 + (m11 - m10) * tx;
    return top + (bot - top) * ty;
}

// The two mesh rows' interpolated values stay in registers while the rows of a
// thread lie between the same centres, so a pixel costs a subtraction, a fused
// multiply-add and its store; converting four FP64 mesh values per pixel took 422 us
// on a 9576 x 6388 map (the FP64 pipe does two conversions per clock and SM), this 53 us.
constexpr int INTERP_ROWS = 16;

__global__ void __launch_bounds__(256) interp_kernel(BgArgs a) {
    const int x0 = (blockIdx.x * 256 + threadIdx.x) * 4;
    if (x0 >= a.pitch) return;
    int ix[4];
    float tx[4], top[4], dif[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        axis_weight(min(x0 + k, a.w - 1), a.w, a.box, a.nx, ix[k], tx[k]);
        top[k] = dif[k] = 0.0f;
    }
    const int jx = a.nx > 1 ? 1 : 0, jy = a.ny > 1 ? a.nx : 0;
    int last = -1;
    for (int yb = blockIdx.y; yb * INTERP_ROWS < a.h; yb += gridDim.y)
    for (int y = yb * INTERP_ROWS, y1 = min(y + INTERP_ROWS, a.h); y < y1; y++) {
        int iy;
        float ty;
        axis_weight(y, a.h, a.box, a.ny, iy, ty);
        if (iy != last) {
            last = iy;
            const float* r0 = a.meshf + (long)iy * a.nx;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const float m00 = r0[ix[k]], m01 = r0[ix[k] + jx], m10 = r0[jy + ix[k]], m11 = r0[jy + ix[k] + jx];
                top[k] = m00 + (m01 - m00) * tx[k];
                dif[k] = m10 + (m11 - m10) * tx[k] - top[k];
            }
        }
        float o[4];
#pragma unroll
        for (int k = 0; k < 4; k++) o[k] = x0 + k < a.w ? top[k] + dif[k] * ty : 0.0f;
        *reinterpret_cast<float4*>(a.map + (long)y * a.pitch + x0) = make_float4(o[0], o[1], o[2], o[3]);
    }
}

template <int NPL>
void launch_box_medians(const BgArgs& a, cudaStream_t s) {
    box_median_kernel<NPL><<<a.nx * a.ny, BOX_THREADS, 0, s>>>(a);
}

// Where a call's scratch lies (bytes from its start): the raw mesh first, then the fill
// value, the mesh in FP32 and the count of cells to fill.
struct BgScratch {
    size_t fill, meshf, missing, bytes;
};
__host__ inline BgScratch bg_scratch(size_t ncell) {
    BgScratch s;
    s.fill = ncell * sizeof(double);
    s.meshf = s.fill + sizeof(double);
    s.missing = s.meshf + ncell * sizeof(float);
    s.bytes = s.missing + sizeof(int);
    return s;
}

}  // namespace

extern "C" int argus_background(argus_ctx* ctx, const float* img, const uint8_t* flags, argus_shape shape,
                                int box, int filt, float min_frac, double* mesh, float* map, argus_stream stream) {
    if (!ctx || !img || !mesh || box < 8 || box > 64 || filt < 1 || filt > 7 || (filt & 1) == 0 ||
        !(min_frac >= 0.0f && min_frac <= 1.0f))
        return ARGUS_ERR_ARG;
    int st = argus_check_shape(shape, ctx->max_pixels);
    if (st) return st;
    if (argus_check_ptr16(img) || (flags && argus_check_ptr16(flags)) || (map && argus_check_ptr16(map)) ||
        ((uintptr_t)mesh & 7u))
        return ARGUS_ERR_ALIGN;
    const int nx = (shape.w + box - 1) / box, ny = (shape.h + box - 1) / box;
    // scratch in the detection label buffer: a frame that fits the context leaves room (pitch >= 8 nx and
    // h >= ny, so at least 32 bytes for each box's 12)
    const BgScratch sc = bg_scratch((size_t)nx * ny);
    if (ny > 65535 || sc.bytes > ctx->max_pixels * sizeof(int)) return ARGUS_ERR_ARG;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return ARGUS_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    BgArgs a;
    a.img = img; a.flags = flags; a.mesh = mesh; a.map = map; a.pitch = shape.pitch;
    a.w = shape.w; a.h = shape.h; a.box = box; a.filt = filt; a.nx = nx; a.ny = ny; a.min_frac = min_frac;
    char* scratch = reinterpret_cast<char*>(ctx->label);
    a.raw = reinterpret_cast<double*>(scratch);
    a.fill = reinterpret_cast<double*>(scratch + sc.fill);
    a.meshf = reinterpret_cast<float*>(scratch + sc.meshf);
    a.missing = reinterpret_cast<int*>(scratch + sc.missing);
    if (cudaMemsetAsync(a.missing, 0, sizeof(int), s) != cudaSuccess) return ARGUS_ERR_CUDA;
    const int npl = (box * box + BOX_THREADS - 1) / BOX_THREADS;   // keys per thread: the smallest compiled bound
    if (npl <= 2) launch_box_medians<2>(a, s);
    else if (npl <= 8) launch_box_medians<8>(a, s);
    else if (npl <= 18) launch_box_medians<18>(a, s);
    else launch_box_medians<32>(a, s);
    mesh_filter_kernel<<<(nx * ny + 255) / 256, 256, 0, s>>>(a);
    mesh_fill_kernel<<<1, FILL_THREADS, 0, s>>>(a); argus_count_launch(3);
    if (map) {
        const int gx = (int)((shape.pitch / 4 + 255) / 256);
        const int gy = min((shape.h + INTERP_ROWS - 1) / INTERP_ROWS, 65535);
        interp_kernel<<<dim3(gx, gy), 256, 0, s>>>(a); argus_count_launch(1);
    }
    return argus_launch_status();
}
