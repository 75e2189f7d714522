// K2: sigma-clipped mean coadd of a stack of raw frames with per-frame
// sub-pixel shifts (paper Sec. 4.1.3, deep coaddition of 30 x 30 s frames into
// a 15-minute coadd; the clipped mean stands in for the matched filter there),
// with calibration fused in.
//
// One thread per output pixel of a 31 x 8 tile.  Per frame, the raw window the
// tile needs is loaded once, coalesced, calibrated and interpolated along x into
// shared memory.  The frame loop is unrolled to the compile-time stack bound NMAX
// so every per-frame sample lives in a register at a static index: invalid or
// absent frames hold +inf and sort to the end.  A merge-exchange network sorts the
// samples; because rejection |v - c| > kappa*s keeps a value-closed set, the
// survivors stay one contiguous range [lo, hi) of the sorted array.
// Traffic: 2 bytes per frame plus 9 bytes of calibration per pixel in, 9 out;
// the instructions per sample bound it (clipping passes, sort, staging).
#include "argus_internal.cuh"

#include <utility>

namespace {

struct CoaddArgs {
    const uint16_t* raw;
    const float* shifts;
    const float* dark;
    const float* flat;
    const uint8_t* bpm;
    float* coadd;
    float* var;
    uint8_t* n_used;
    long pitch, frame_stride;
    int w, h, nf, bias, sat, max_iter;
    float gain, rn2, kappa;
};

// Batcher's merge exchange (odd-even merge sort) of N values: 191 compare-exchanges
// for N = 32 (a bitonic network has 240), the pairs listed at compile time so
// that every index is static.
template <int N> struct SortNet {
    unsigned char a[N * 16], b[N * 16];
    int n;
};
template <int N> constexpr SortNet<N> make_sort_net() {
    SortNet<N> t{};
    for (int p = 1; p < N; p *= 2)
        for (int k = p; k >= 1; k /= 2)
            for (int j = k % p; j + k < N; j += 2 * k)
                for (int i = 0; i < k && i + j + k < N; i++)
                    if ((i + j) / (2 * p) == (i + j + k) / (2 * p)) {
                        t.a[t.n] = (unsigned char)(i + j);
                        t.b[t.n++] = (unsigned char)(i + j + k);
                    }
    return t;
}
template <int N> struct SortPairs { static constexpr SortNet<N> net = make_sort_net<N>(); };
template <int I, int J, int N>
__device__ __forceinline__ void exchange(float (&s)[N]) {
    const float a = s[I], b = s[J];
    s[I] = fminf(a, b);
    s[J] = fmaxf(a, b);
}
template <int N, int... E>
__device__ __forceinline__ void sort_list(float (&s)[N], std::integer_sequence<int, E...>) {
    (exchange<SortPairs<N>::net.a[E], SortPairs<N>::net.b[E], N>(s), ...);
}
template <int N>
__device__ __forceinline__ void sort_values(float (&s)[N]) {
    sort_list(s, std::make_integer_sequence<int, SortPairs<N>::net.n>());
}

// One CTA per 31 x 8 output tile.  Per tile:
//
// Phase 0: the calibration constants (the reciprocal of the flat, or NaN where
// the pixel is unusable -- outside the frame, flagged bad, flat not positive
// and finite -- and the dark) of the union of the frames' windows into shared
// memory, once: frames share their pixels' calibration, and their windows
// differ only by the integer parts of the shifts.  When that union exceeds
// UCAP pixels (shifts spread by more than 4 px) each frame's window reads its
// constants from global memory instead.
//
// Phase 1: a warp per frame: the frame's 32 x 9 window of raw pixels -- at the
// frame's integer offset -- row by row, one pixel per lane, calibrated (the flat
// enters through its correctly rounded reciprocal, within 1 ulp of the quotient)
// and interpolated along x with the next lane's pixel: the row lerp of the value
// (NaN where a needed pixel is unusable) and the same for the variance by the
// squared weights.  A row lerp serves the output rows above and below it, and
// everything about the frame is the same for the whole warp.  Tiles are 31 wide
// so that the 32 lanes hold every neighbour.
//
// Phase 2: each thread interpolates its samples along y from two shared values
// per frame, sorts them in registers and writes the sorted column to shared
// memory.  A clipping pass takes the median from two slots of it, the sums of
// v - c and (v - c)^2 over the range from the registers, in ascending order
// (values outside the range are skipped), and the rejected samples by scanning
// inward from both ends (the rejected set is a prefix below the median and a
// suffix above it, because the rounded distance to the median is monotone in the
// sample).  The variance of the mean then sums the variances of the samples
// inside the surviving range, compensated.
//
// 30 frames of 9576 x 6388: 11.5 ms (4,340 thread instructions per pixel of a
// 32-frame stack: staging and samples 55 a frame, sort and set-up 820, clipping 920;
// issue slots 58 % busy with the 16 warps that 105 KB a CTA leave room for), against
// 18.7 ms with the window staged pixel by pixel over all threads, four-neighbour
// samples, a bitonic sort and clipping sums from shared memory.
constexpr int CTX = 31, CTY = 8, CWX = 32, CWY = CTY + 1, CWN = CWX * CWY;
constexpr int CT = 32 * CTY;                   // threads (one per output pixel of the tile; lane 31 has none)
constexpr int UCAP = 512;                      // union window capacity (pixels): shift spreads up to 4 px
constexpr float FMAXF = 3.402823466e38f;

__device__ __forceinline__ float qnan() { return __int_as_float(0x7fffffff); }

// Median of the sorted range [lo, hi) of one thread's column of samples
// (slot i at col[i * CT]); the mean of the two middle values for even counts.
__device__ __forceinline__ float median_col(const float* col, int lo, int hi) {
    const int n = hi - lo;
    const float a = col[(lo + (n - 1) / 2) * CT], b = col[(lo + n / 2) * CT];
    return (n & 1) ? b : 0.5f * (a + b);
}

// Calibration constants of frame pixel (gx, gy): (1 / flat, dark), with NaN
// in place of 1 / flat when the pixel is unusable.
__device__ __forceinline__ float2 calib_const(const CoaddArgs& a, int gx, int gy) {
    float2 c = make_float2(qnan(), 0.0f);
    if (gx >= 0 && gy >= 0 && gx < a.w && gy < a.h) {
        const long p = (long)gy * a.pitch + gx;
        const float fl = a.flat ? __ldg(a.flat + p) : 1.0f;
        const bool bad = a.bpm && __ldg(a.bpm + p);
        if (!bad && fl > 0.0f && fl <= FMAXF) c.x = __frcp_rn(fl);
        c.y = a.dark ? __ldg(a.dark + p) : 0.0f;
    }
    return c;
}

// Calibrated (value, variance) of one raw pixel given its constants, without a
// branch: the value is NaN where unusable (the variance then means nothing).
__device__ __forceinline__ float2 calib_pair(const CoaddArgs& a, int raw, float2 c) {
    const float ng = (float)(raw - a.bias) * a.gain;
    const float cv = (ng - c.y) * c.x;
    const bool ok = (raw < a.sat) & (fabsf(cv) <= FMAXF);   // false for NaN constants
    return make_float2(ok ? cv : qnan(), (fmaxf(ng, 0.0f) + a.rn2) * (c.x * c.x));
}

// One axis of a frame's shift: its integer part, its fraction f, and the squared weights
// (1 - f)^2 and f^2 of the variances, each rounded once (their errors are the same for every pixel of
// the frame, so they count: with squares of rounded FP32 differences the rms error of 3 frames'
// variance was 1.00e-7 of it, now 0.91e-7; 9 to 64 frames 0.80e-7 to 0.87e-7 either way).  A
// window that starts
// `size` pixels (the frame's extent along the axis) past a tile's own place, or the window's
// own extent more than that before it, meets no pixel of the frame from any tile, so larger shifts are
// held there; so is one that is not a number.  Window coordinates and the windows' union
// then stay in range whatever the shifts are.
struct ShiftPart { int whole; float frac, w0, w1; };
__host__ __device__ __forceinline__ ShiftPart split_shift(float shift, int size) {
    const double d = shift, fl = floor(d);
    const float f = (float)(d - fl);
    return {(int)fmin(fmax(fl, -(double)size - CWX), (double)size), f, (float)((1.0 - f) * (1.0 - f)), (float)((double)f * f)};
}
// Whether the union of windows whose integer shifts span dx and dy pixels fits the shared table.
__host__ __device__ __forceinline__ bool union_fits(int dx, int dy) {
    return ((long)CWX + dx) * ((long)CWY + dy) <= UCAP;
}

// The raw pixels of column gx, rows gy .. gy + 8 of frame f (clamped to the frame).
__device__ __forceinline__ void load_window(const CoaddArgs& a, int f, int gx, int gy, int (&raw)[CWY]) {
    const uint16_t* src = a.raw + (long)f * a.frame_stride + min(max(gx, 0), a.w - 1);
    if (gy >= 0 && gy + CWY <= a.h) {      // the same for the whole warp
        src += (long)gy * a.pitch;
#pragma unroll
        for (int r = 0; r < CWY; r++, src += a.pitch) raw[r] = __ldg(src);
        return;
    }
#pragma unroll
    for (int r = 0; r < CWY; r++) raw[r] = __ldg(src + (long)min(max(gy + r, 0), a.h - 1) * a.pitch);
}

// Four CTAs an SM for stacks of up to 8: such a tile is mostly waiting (calibration constants, barriers,
// stores), and at the 80 registers a thread that the compiler takes otherwise three fit (3 frames
// of 9576 x 6388: 2.22 ms, now 1.85; five CTAs of 48 registers 1.87).
template <int NMAX>
__global__ void __launch_bounds__(CT, NMAX <= 8 ? 4 : NMAX <= 32 ? 2 : 1) coadd_kernel(CoaddArgs a) {
    extern __shared__ float4 coadd_smem[];
    float* wv = reinterpret_cast<float*>(coadd_smem);            // [nf][CWN] row-interpolated values
    float* wq = wv + a.nf * CWN;                                 // [nf][CWN] and variances
    float* ss = wq + a.nf * CWN;                                 // [NMAX][CT] sorted samples, a column per thread
    float2* ucal = reinterpret_cast<float2*>(ss + NMAX * CT);    // [UCAP] union calibration window
    __shared__ int s_ix[NMAX], s_iy[NMAX];
    __shared__ float4 s_x[NMAX];           // fx, (1 - fx)^2, fx^2
    __shared__ float4 s_y[NMAX];           // fy, (1 - fy)^2, fy^2, offset of the next row (0 when it has no weight)
    __shared__ int s_umin[2], s_uwh[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) { s_umin[0] = s_umin[1] = 1 << 30; s_uwh[0] = s_uwh[1] = -(1 << 30); }
    __syncthreads();
    for (int f = tid; f < a.nf; f += blockDim.x) {
        const ShiftPart sx = split_shift(a.shifts[2 * f], a.w), sy = split_shift(a.shifts[2 * f + 1], a.h);
        const int ix = sx.whole, iy = sy.whole;
        atomicMin(&s_umin[0], ix); atomicMin(&s_umin[1], iy);
        atomicMax(&s_uwh[0], ix); atomicMax(&s_uwh[1], iy);
        s_ix[f] = ix;
        s_iy[f] = iy;
        s_x[f] = make_float4(sx.frac, sx.w0, sx.w1, 0.0f);
        s_y[f] = make_float4(sy.frac, sy.w0, sy.w1, __int_as_float(sy.frac > 0.0f ? CWX : 0));
    }
    __syncthreads();
    const int ixmin = s_umin[0], iymin = s_umin[1];
    const int UW = CWX + (s_uwh[0] - ixmin), UH = CWY + (s_uwh[1] - iymin);
    const bool uni = union_fits(s_uwh[0] - ixmin, s_uwh[1] - iymin);   // the same for every CTA
    const int ntx = (a.w + CTX - 1) / CTX, nty = (a.h + CTY - 1) / CTY;
    const int o = warp * CWX + lane;       // output row `warp`, column `lane`
    float* col = ss + tid;
    for (int tile = blockIdx.x; tile < ntx * nty; tile += gridDim.x) {
        const int tx0 = (tile % ntx) * CTX, ty0 = (tile / ntx) * CTY;
        const int x = tx0 + lane, y = ty0 + warp;
        // a warp's next frame is loaded while it works on this one; pixels off the frame read the
        // nearest one and are unusable through their constants
        int raw[CWY];
        if (warp < a.nf) load_window(a, warp, tx0 + s_ix[warp] + lane, ty0 + s_iy[warp], raw);
        __syncthreads();   // the previous tile's windows are consumed
        if (uni) {
            for (int e = tid; e < UW * UH; e += blockDim.x) {
                const int uy = e / UW, ux = e - uy * UW;
                ucal[e] = calib_const(a, tx0 + ixmin + ux, ty0 + iymin + uy);
            }
            __syncthreads();
        }
        for (int f = warp; f < a.nf; f += CTY) {
            const int gx = tx0 + s_ix[f] + lane, gy = ty0 + s_iy[f];
            float2 c[CWY];
            if (uni) {
                const float2* uc = ucal + (s_iy[f] - iymin) * UW + (s_ix[f] - ixmin) + lane;
#pragma unroll
                for (int r = 0; r < CWY; r++) c[r] = uc[r * UW];
            } else {
#pragma unroll
                for (int r = 0; r < CWY; r++) c[r] = calib_const(a, gx, gy + r);
            }
            float2 p[CWY];
#pragma unroll
            for (int r = 0; r < CWY; r++) p[r] = calib_pair(a, raw[r], c[r]);
            const int fn = f + CTY;
            if (fn < a.nf) load_window(a, fn, tx0 + s_ix[fn] + lane, ty0 + s_iy[fn], raw);
            const float4 wx = s_x[f];
            const float fx = wx.x, w0 = wx.y, w1 = wx.z;
            float* dv = wv + f * CWN + lane;
            float* dq = wq + f * CWN + lane;
            if (fx > 0.0f) {
#pragma unroll
                for (int r = 0; r < CWY; r++) {
                    const float nv = __shfl_down_sync(0xffffffffu, p[r].x, 1), nq = __shfl_down_sync(0xffffffffu, p[r].y, 1);
                    dv[r * CWX] = __fmaf_rn(fx, __fsub_rn(nv, p[r].x), p[r].x);
                    dq[r * CWX] = w0 * p[r].y + w1 * nq;
                }
            } else {
#pragma unroll
                for (int r = 0; r < CWY; r++) {
                    dv[r * CWX] = p[r].x;
                    dq[r * CWX] = p[r].y;
                }
            }
        }
        __syncthreads();
        if (lane >= CTX || x >= a.w || y >= a.h) continue;
        float s[NMAX];
        int n = 0;
        const float* pv = wv + o;
#pragma unroll
        for (int fi = 0; fi < NMAX; fi++) {
            s[fi] = __int_as_float(0x7f800000);      // +inf: absent or invalid
            if (fi < a.nf) {
                const float4 fy = s_y[fi];
                const float top = pv[fi * CWN], bot = pv[fi * CWN + __float_as_int(fy.w)];
                const float v = __fmaf_rn(fy.x, __fsub_rn(bot, top), top);
                const bool ok = fabsf(v) <= FMAXF;
                s[fi] = ok ? v : s[fi];
                n += ok ? 1 : 0;
            }
        }
        sort_values(s);
#pragma unroll
        for (int i = 0; i < NMAX; i++) col[i * CT] = s[i];
        int lo = 0, hi = n;
        float last_s1 = 0.0f;   // sum of v - median over [lo, hi) when the last pass kept every sample
        bool have_s1 = false;
        // the sums over [lo, hi) about c, in ascending order
        const auto sums = [&](float c, float& s1, float& s2) {
            const unsigned long long in = (hi < 64 ? (1ull << hi) - 1ull : ~0ull) & ~((1ull << lo) - 1ull);
            s1 = s2 = 0.0f;
#pragma unroll
            for (int i = 0; i < NMAX; i++)
                if ((in >> i) & 1ull) {
                    const float d = s[i] - c;
                    s1 += d;
                    s2 = fmaf(d, d, s2);
                }
        };
        for (int it = 0; it < a.max_iter && hi > lo; it++) {
            const int cnt = hi - lo;
            const float c = median_col(col, lo, hi);
            // mean and spread in one pass over the range, about the median (the sums of
            // v - c and (v - c)^2; the median lies inside the samples, so the difference
            // of the second sum and the squared first one does not cancel)
            float s1, s2;
            sums(c, s1, s2);
            const float d1 = s1 / (float)cnt;
            const float ks = a.kappa * sqrtf(fmaxf(s2 / (float)cnt - d1 * d1, 0.0f));
            int nlo = 0, nhi = 0;
            while (lo + nlo < hi) {
                const float v = col[(lo + nlo) * CT];
                if (!(v < c && fabsf(v - c) > ks)) break;
                nlo++;
            }
            while (hi - 1 - nhi >= lo + nlo) {
                const float v = col[(hi - 1 - nhi) * CT];
                if (!(v >= c && fabsf(v - c) > ks)) break;
                nhi++;
            }
            if (nlo + nhi == 0) {
                last_s1 = s1;
                have_s1 = true;
                break;
            }
            if (nlo + nhi == cnt) break;
            lo += nlo;
            hi -= nhi;
        }
        const long p = (long)y * a.pitch + x;
        if (hi <= lo) {
            a.coadd[p] = 0.0f;
            a.var[p] = 0.0f;
            a.n_used[p] = 0;
            continue;
        }
        const int cnt = hi - lo;
        const float c = median_col(col, lo, hi);
        const float vlo = col[lo * CT], vhi = col[(hi - 1) * CT];
        float sd = last_s1;   // the converged pass's sum over the same range about the same median
        if (!have_s1) {
            float s2;
            sums(c, sd, s2);
        }
        // the survivors' variances (Kahan's compensated sum; the library is not built with fast-math)
        float sv = 0.0f, se = 0.0f;
        const float* pq = wq + o;
#pragma unroll 6
        for (int fi = 0; fi < a.nf; fi++) {
            const float4 fy = s_y[fi];
            const int dn = __float_as_int(fy.w);
            const float top = pv[fi * CWN], bot = pv[fi * CWN + dn];
            const float v = __fmaf_rn(fy.x, __fsub_rn(bot, top), top);
            const float q = fy.y * pq[fi * CWN] + fy.z * pq[fi * CWN + dn];
            if (v >= vlo && v <= vhi) {                // NaN and infinite samples lie outside
                const float t = q - se, u = sv + t;
                se = (u - sv) - t;
                sv = u;
            }
        }
        a.coadd[p] = c + sd / (float)cnt;
        a.var[p] = sv / ((float)cnt * (float)cnt);
        a.n_used[p] = (uint8_t)cnt;
    }
}

template <int NMAX>
int launch(const CoaddArgs& a, int sms, cudaStream_t st) {
    const size_t smem = ((size_t)a.nf * CWN * 2 + (size_t)NMAX * CT + (size_t)UCAP * 2) * sizeof(float);
    if (cudaFuncSetAttribute(coadd_kernel<NMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess ||
        cudaFuncSetAttribute(coadd_kernel<NMAX>, cudaFuncAttributePreferredSharedMemoryCarveout, 100) != cudaSuccess)
        return ARGUS_ERR_CUDA;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, coadd_kernel<NMAX>, CT, smem) != cudaSuccess ||
        per_sm < 1)
        return ARGUS_ERR_CUDA;
    const long tiles = (long)((a.w + CTX - 1) / CTX) * ((a.h + CTY - 1) / CTY);
    long blocks = tiles;
    if (blocks > (long)sms * per_sm) blocks = (long)sms * per_sm;
    coadd_kernel<NMAX><<<(unsigned)blocks, CT, smem, st>>>(a); argus_count_launch(1);
    return argus_launch_status();
}

}  // namespace

extern "C" int argus_coadd(argus_ctx* ctx, const uint16_t* raw_stack, int n, argus_shape shape,
                           const float* shifts_xy, const argus_calib* calib, float kappa, int max_iter,
                           float* coadd, float* var, uint8_t* n_used, argus_stream stream) {
    if (!ctx || !raw_stack || !shifts_xy || !calib || !coadd || !var || !n_used) return ARGUS_ERR_ARG;
    if (n < 1 || n > ARGUS_MAX_FRAMES || max_iter < 0 || !(kappa > 0.0f)) return ARGUS_ERR_ARG;
    if (calib->bias_frame) return ARGUS_ERR_UNSUPPORTED;
    int rc = argus_check_shape(shape, ctx->max_pixels);
    if (rc) return rc;
    const void* ps[] = {raw_stack, coadd, var, n_used, calib->dark, calib->flat, calib->bpm};
    for (const void* p : ps)
        if (p && argus_check_ptr16(p)) return ARGUS_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return ARGUS_ERR_CUDA;
    CoaddArgs a;
    a.raw = raw_stack; a.shifts = shifts_xy; a.dark = calib->dark; a.flat = calib->flat; a.bpm = calib->bpm;
    a.coadd = coadd; a.var = var; a.n_used = n_used; a.pitch = shape.pitch;
    a.frame_stride = shape.pitch * (long)shape.h; a.w = shape.w; a.h = shape.h; a.nf = n;
    a.bias = calib->bias_scalar; a.sat = calib->sat; a.max_iter = max_iter; a.gain = calib->gain;
    a.rn2 = calib->read_noise * calib->read_noise; a.kappa = kappa;
    cudaStream_t st = (cudaStream_t)stream;
    if (n <= 8) return launch<8>(a, ctx->num_sms, st);
    if (n <= 16) return launch<16>(a, ctx->num_sms, st);
    if (n <= 32) return launch<32>(a, ctx->num_sms, st);
    return launch<64>(a, ctx->num_sms, st);
}
