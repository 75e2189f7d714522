// K9 forward on the tensor cores: the learned kernel surrogate's whole forward
// pass (1x1 conv 2 -> 32, four 7x7 'same' 32 -> 32 convolutions with ReLU,
// 1x1 conv 32 -> 1, output / 441) in one persistent kernel, the four 7x7
// convolutions as implicit GEMMs on tcgen05 (kind::f16: BF16 operands, FP32
// accumulation in TMEM).  The paper has no learned kernel; this is the learned
// alternative to its least-squares PSF-matching kernel (Sec. 4.2).
//
// Implicit GEMM.  A stamp's activations sit in shared memory zero padded to 27
// rows (21 + 6) of 32 pixels (27 used) and flattened: plane pixel P = 32 row + col.
// The kernel columns kx go into N: with A = 128 consecutive plane pixels (four
// image rows) at row offset ky,
//   T[P][(kx, o)] = sum_{ky, i} A[P + 32 ky][i] W[ky][kx][i][o],   N = 7 x 32 = 224,
//   out[x][o] = sum_kx T[x + kx][(kx, o)],
// and a warp's 32 TMEM lanes are one image row, so the last sum is six lane shifts in
// the epilogue.  An MMA of N = 32 takes 47 clocks of the tensor pipe where its share of
// the dense rate is 16; one of N = 224 takes its 112.  Per layer 6 tiles (rows 4 t .. 4 t
// + 3; the last holds row 20) x 7 ky x 2 halves of the 32 input channels x 2 parts = 168
// MMAs, 18.8 k clocks, against 980 of N = 32 with every tap an MMA of its own, 46 k.
//
// Precision.  Activations are split into BF16 hi + lo (v = hi + lo + e, |e| <=
// 2^-17 |v|) and each runs against the BF16 weights, so the layer is the FP32 layer
// to within FP32-level rounding: the same weights as the SIMT BF16 path,
// activations to ~16 significant bits instead of BF16's 8.
//
// Layouts.  Operand planes [hi|lo][chunk of 8 channels][864 plane pixels][8]
// (BF16, 16 bytes per pixel and chunk): a K-major core matrix is 8 consecutive
// pixels of one chunk (128 contiguous bytes), LBO = one plane (the next 8
// channels), SBO = 128 bytes.  (The last tile's unused rows read on into the next
// plane or the weights.)  Weights are packed once per call into
// [layer][ky][chunk][kx * 32 + o][8] (14 KB per ky, LBO 3,584, SBO 128); a layer's seven
// are brought in by bulk copies in two groups, the next layer's first three when the last
// tile is done with them, the other four after it.  (A wait or a commit costs the issuing
// thread 200 to 500 clocks, so seven of each per layer cost more than the overlap gained.)
//
// Roles (576 threads, one CTA per SM): warp 0 allocates TMEM and one lane issues the
// MMAs; warp 1 lane 0 streams the weights; 16 warps, four per quarter of the TMEM lanes,
// take 8 of the 32 channels each: they write layer 1 into the planes and then, per tile,
// read their columns of the accumulator (two buffers of 224 columns), shift and sum, add
// the bias, apply ReLU and write the next layer's planes in place -- tile t's rows once
// tile t + 1's MMAs have completed, the last that read them -- optionally the FP32
// activations for the backward pass, and after the last layer the 1x1 output (the four
// channel groups' parts through shared memory).  A tile's buffer is free for the tile
// after next once it is read, so that reading sets the pace unless it takes less than a
// tile's MMAs.  The MMAs of the next layer's tile t wait only for the rows they read
// (tiles up to t + 1), so layers follow one another without a gap.  Every wait is
// bounded; a timeout latches ARGUS_ERR_TIMEOUT and all roles stop.
//
// 400 stamps: 150 us (46 us an image and SM, three rounds), against 406 us for one MMA of
// N = 32 per tap and two CTAs an SM.  With the MMAs issued from a branch of one lane an
// image took 61 us whatever N was (see mma_bf16_warp).
//
// The data gradient of each 7x7 layer is the same implicit GEMM with the
// layer's kernel transposed and flipped: the gradient planes dz (BF16 hi + lo)
// against W'[ky][kx][o][i] = W[6 - ky][6 - kx][i][o], one layer per launch.
#include <cuda_bf16.h>

#include "cnn_net.cuh"

namespace {

using namespace cnn_net;

constexpr int WP = 32;                    // plane row pitch: one warp of lanes
constexpr int NPP = (S + KS - 1) * WP;    // 864 plane pixels
constexpr int PLANE = NPP * 16;           // one 8-channel chunk plane (BF16): 13,824 bytes
constexpr int SETB = (C / 8) * PLANE;     // one operand set (hi or lo): 55,296 bytes
constexpr int MT = 6;                     // M tiles of four image rows
constexpr int NN = KS * C;                // 224 accumulator columns of a tile
constexpr int KYB = (C / 8) * NN * 16;    // one kernel row's B operand: 14,336 bytes
constexpr int KYA = 3;                    // kernel rows of a layer's first weight group (the second holds the rest)
constexpr int NG = 4, GC = C / NG;        // channel groups of the epilogue, channels of each
constexpr int NEPI = 4 * NG;              // epilogue warps
constexpr int NTHR = 64 + 32 * NEPI;
constexpr uint32_t TMEM_COLS = 512;       // two accumulator buffers, 256 columns apart
// the last tile's rows reach 3 plane rows past the planes: into the next chunk, or the ring
static_assert((4 * (MT - 1) + KS - 1) * WP + 128 <= NPP + 3 * WP && 3 * WP * 16 <= KYB, "tile reads stay inside the block");

struct CnnTcShared {
    alignas(128) uint8_t act[2][SETB];    // operand planes: [hi | lo][chunk][pixel][8 channels]
    alignas(128) uint8_t wb[KS][KYB];     // a layer's per-ky B operands
    float w1[2 * C], b1[C], bc[4][C], w6[C], b6;
    float ypart[2][NG][128];              // channel groups' parts of a tile's outputs
    uint64_t wfull[2], wempty[2], wrote[MT], accfull[MT], accempty[2], yfull[2], drain;
    uint32_t tmem;
    int abort;
};
static_assert(sizeof(CnnTcShared) + 1024 <= 228 * 1024, "one CTA per SM");

// The 8 channels of chunk ic of plane pixel P as BF16 hi and lo parts into both operand sets.
__device__ __forceinline__ void store_chunk(CnnTcShared& sh, int ic, int P, const float (&h)[GC]) {
    split_chunk(h, sh.act[0] + ic * PLANE + P * 16, sh.act[1] + ic * PLANE + P * 16);
}

// Packs the BF16 weights W[l][ky][kx][i][o] of the four 7x7 layers into the
// B-operand layout [l][ky][i / 8][kx 32 + o][i % 8].
__global__ void cnn_pack_tc_kernel(const __nv_bfloat16* w, __nv_bfloat16* wp) {
    const long tot = 4L * NTAP * C * C;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < tot; e += (long)gridDim.x * blockDim.x) {
        const int j = (int)(e & 7), n = (int)((e >> 3) % NN);
        const long r = (e >> 3) / NN;                        // (l, ky, chunk)
        const int ic = (int)(r & 3), ky = (int)((r >> 2) % KS), l = (int)((r >> 2) / KS);
        const int kx = n / C, o = n % C;
        wp[e] = w[off_w(l) + ((long)(ky * KS + kx) * C + ic * 8 + j) * C + o];
    }
}

// Packs the BF16 weights of 7x7 layer l for its data gradient: the transposed, flipped
// kernel W'[ky][kx][o][i] = W[6 - ky][6 - kx][i][o] in the B-operand layout
// [ky][o / 8][kx 32 + i][o % 8] (N the layer's input channels, K its output channels).
__global__ void cnn_pack_dgrad_tc_kernel(const __nv_bfloat16* w, __nv_bfloat16* wp, int l) {
    const long tot = (long)NTAP * C * C;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < tot; e += (long)gridDim.x * blockDim.x) {
        const int j = (int)(e & 7), n = (int)((e >> 3) % NN);
        const long r = (e >> 3) / NN;
        const int oc = (int)(r & 3), ky = (int)(r >> 2), kx = n / C, i = n % C;
        const int ft = (KS - 1 - ky) * KS + (KS - 1 - kx);
        wp[e] = w[off_w(l) + ((long)ft * C + i) * C + oc * 8 + j];
    }
}

struct CnnTcArgs {
    const float* x;                 // forward: [n][441][2]
    const __nv_bfloat16* w;         // forward: the parameter vector
    float* y;                       // forward: [n][441]
    float* acts;                    // forward, optional: h1 .. h5 at acts + l * lstride, [n][441][32] FP32
    long lstride;
    const float* dh_out;            // gradient: [n][441][32]
    const float* h_out;
    float* dh_in;
    const uint8_t* wpack;
    int n;
    int* status;
};

// A warp's sum over the kernel columns for one tile: lane x gets out[x][o] = sum_kx
// T[x + kx][(kx, o)] of its 8 channels, tl the accumulator's first of them (its lanes are
// one image row; lanes past 25 wrap and mean nothing).  The loads are all in flight at once.
__device__ __forceinline__ void shift_sum(uint32_t tl, float (&h)[GC]) {
    uint32_t v[KS][GC];
#pragma unroll
    for (int kx = 0; kx < KS; kx++) tc::tmem_ld8_nowait(tl + (uint32_t)(kx * C), v[kx]);
    tc::tmem_wait_ld();
#pragma unroll
    for (int kx = 0; kx < KS; kx++) tc::tmem_use8(v[kx]);
#pragma unroll
    for (int kx = 0; kx < KS; kx++)
#pragma unroll
        for (int o = 0; o < GC; o++) {
            const float f = __uint_as_float(v[kx][o]);
            h[o] = kx ? h[o] + __shfl_down_sync(0xffffffffu, f, kx) : f;
        }
}

// The four 7x7 layers of the forward (BWD = false), or one layer's data gradient:
// dz = dh_out (h_out > 0) and
//   dh_in[y][x][i] = sum_{ky,kx,o} W[ky][kx][i][o] dz[y - ky + 3][x - kx + 3][o]
//                  = sum_{ky,kx,o} W'[ky][kx][o][i] dz[y + ky - 3][x + kx - 3][o].
template <bool BWD>
__global__ void __launch_bounds__(NTHR, 1) cnn_tc_kernel(CnnTcArgs a) {
    constexpr int NL = BWD ? 1 : 4;
    extern __shared__ __align__(1024) uint8_t cnn_tc_smem[];
    CnnTcShared& sh = *reinterpret_cast<CnnTcShared*>(cnn_tc_smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (!BWD) {
        for (int e = tid; e < 2 * C; e += NTHR) sh.w1[e] = __bfloat162float(a.w[OFF_W1 + e]);
        for (int e = tid; e < C; e += NTHR) {
            sh.b1[e] = __bfloat162float(a.w[OFF_B1 + e]);
            sh.w6[e] = __bfloat162float(a.w[OFF_W6 + e]);
        }
        for (int e = tid; e < 4 * C; e += NTHR) sh.bc[e / C][e % C] = __bfloat162float(a.w[off_b(e / C) + e % C]);
        if (tid == 0) sh.b6 = __bfloat162float(a.w[OFF_B6]);
    }
    // both operand sets zeroed once: the padding stays zero, interiors are rewritten per layer
    for (int e = tid; e < 2 * SETB / 16; e += NTHR) reinterpret_cast<uint4*>(sh.act[0])[e] = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        for (int g = 0; g < 2; g++) {
            tc::mbar_init(&sh.wfull[g], 1);
            tc::mbar_init(&sh.wempty[g], 1);
        }
        for (int t = 0; t < MT; t++) {
            tc::mbar_init(&sh.wrote[t], NEPI);
            tc::mbar_init(&sh.accfull[t], 1);
        }
        for (int b = 0; b < 2; b++) {
            tc::mbar_init(&sh.accempty[b], NEPI);
            tc::mbar_init(&sh.yfull[b], 4 * (NG - 1));
        }
        tc::mbar_init(&sh.drain, 1);
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tc::tmem_alloc(&sh.tmem, TMEM_COLS);
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = sh.tmem;

    if (warp == 0) {
        // ---------------- MMA issuer (the whole warp runs it, lane 0 issues)
        const uint32_t el = lane == 0;
        const uint32_t idesc = tc::instr_desc(1, 128, NN);
        const uint64_t a0 = tc::smem_desc(tc::smem_u32(sh.act[0]), PLANE, 128);
        const uint64_t b0 = tc::smem_desc(tc::smem_u32(sh.wb[0]), NN * 16, 128);
        int lay = 0, tile = 0;                           // layers and tiles so far
        bool run = true, any = false;
        for (int img = blockIdx.x; img < a.n && run; img += gridDim.x) {
            for (int l = 0; l < NL && run; l++, lay++) {
#pragma unroll 1
                for (int t = 0; t < MT && run; t++, tile++) {
                    const int b = tile & 1;
                    // the accumulator drained, and the rows this tile reads written (tile t - 1 has
                    // waited for the earlier ones)
                    if ((tile >= 2 && !tc::all_lanes(wait_or_abort(sh, &sh.accempty[b], ((tile >> 1) - 1) & 1, a.status))) ||
                        (t == 0 && !tc::all_lanes(wait_or_abort(sh, &sh.wrote[0], lay & 1, a.status))) ||
                        (t + 1 < MT && !tc::all_lanes(wait_or_abort(sh, &sh.wrote[t + 1], lay & 1, a.status)))) {
                        run = false;
                        break;
                    }
                    tc::fence_after();
                    const uint32_t acc = tmem + (uint32_t)(b * 256);
                    const uint64_t at = a0 + (uint32_t)(4 * t * WP);   // descriptors count in 16 bytes: a plane pixel
#pragma unroll
                    for (int ky = 0; ky < KS; ky++) {
                        if (t == 0 && (ky == 0 || ky == KYA)) {
                            if (run) run = tc::all_lanes(wait_or_abort(sh, &sh.wfull[ky ? 1 : 0], lay & 1, a.status));
                            tc::fence_after();
                        }
                        if (run) {
#pragma unroll
                            for (int kc = 0; kc < 2; kc++)
#pragma unroll
                                for (int hl = 0; hl < 2; hl++)
                                    tc::mma_bf16_warp(acc, at + (uint32_t)(ky * WP + (hl * SETB + 2 * kc * PLANE) / 16),
                                                      b0 + (uint32_t)((ky * KYB + kc * 2 * NN * 16) / 16), idesc,
                                                      (ky | kc | hl) ? 1u : 0u, el);
                            any = true;
                            if (t == MT - 1 && (ky == KYA - 1 || ky == KS - 1)) tc::commit_warp(&sh.wempty[ky == KS - 1 ? 1 : 0], el);
                        }
                    }
                    if (run) tc::commit_warp(&sh.accfull[t], el);
                }
            }
        }
        // every issued MMA lands before TMEM is released
        if (any) {
            tc::commit_warp(&sh.drain, el);
            if (!tc::mbar_wait_bounded(&sh.drain, 0, WAIT_LIMIT)) {
                sh.abort = 1;
                argus_latch(a.status, ARGUS_ERR_TIMEOUT);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- weight producer: a layer's two groups of kernel rows, in the MMA order
        if (lane == 0) {
            int lay = 0, g = 0;                      // group g of layer lay is the next to be asked for
            bool run = true;
            for (int img = blockIdx.x; img < a.n && run; img += gridDim.x)
                for (int l = 0; l < NL && run; l++, lay++)
                    for (g = 0; g < 2; g++) {
                        if (lay && !wait_or_abort(sh, &sh.wempty[g], (lay - 1) & 1, a.status)) { run = false; break; }
                        const int k0 = g ? KYA : 0, k1 = g ? KS : KYA;
                        tc::mbar_arrive_expect_tx(&sh.wfull[g], (uint32_t)((k1 - k0) * KYB));
                        for (int ky = k0; ky < k1; ky++)
                            tc::bulk_g2s(sh.wb[ky], a.wpack + (long)(l * KS + ky) * KYB, KYB, &sh.wfull[g]);
                    }
            // copies in flight land before the CTA exits (the latest phase of each group)
            if (!run) lay--;                         // the loop's step after the break
            for (int q = 0; q < 2; q++) {
                const int ph = run || q >= g ? lay - 1 : lay;     // groups below g of layer lay were asked for
                if (ph >= 0 && !tc::mbar_wait_bounded(&sh.wfull[q], ph & 1, WAIT_LIMIT)) {
                    sh.abort = 1;
                    argus_latch(a.status, ARGUS_ERR_TIMEOUT);
                    break;
                }
            }
        }
        __syncwarp();
    } else {
        // ---------------- first planes, epilogues, output
        const int grp = (warp - 2) >> 2;             // channels 8 grp .. 8 grp + 7, operand chunk grp
        const int lq = warp & 3;                     // the TMEM lane quarter this warp may read: image row 4 t + lq
        const uint32_t tl = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(grp * GC);
        // a condition that one lane waits for
        const auto landed = [&](uint64_t* bar, int parity) {
            bool ok = true;
            if (lane == 0) ok = wait_or_abort(sh, bar, parity & 1, a.status);
            ok = __shfl_sync(0xffffffffu, ok, 0);
            return ok;
        };
        const auto wrote = [&](int t) {
            tc::fence_proxy_async();                 // plane writes visible to the tensor cores
            tc::fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sh.wrote[t]);
        };
        // the group's channels of an image's first planes (layer 1 of the inputs xn, or dz)
        float xn[BWD ? 1 : MT][2];
        const auto fetch = [&](int img) {
            if constexpr (!BWD) {
#pragma unroll
                for (int t = 0; t < MT; t++) {
                    const int row = 4 * t + lq;
                    const bool mine = row < S && lane < S;
                    const float* xp = a.x + ((long)img * NPX + (mine ? row * S + lane : 0)) * 2;
                    xn[t][0] = xp[0];
                    xn[t][1] = xp[1];
                }
            }
        };
        const auto fill = [&](int img) {
#pragma unroll
            for (int t = 0; t < MT; t++) {
                const int row = 4 * t + lq;
                if (row < S && lane < S) {
                    const long p = (long)img * NPX + row * S + lane;
                    float h[GC];
                    if constexpr (BWD) {
                        const float4* go = reinterpret_cast<const float4*>(a.dh_out + p * C + grp * GC);
                        const float4* ho = reinterpret_cast<const float4*>(a.h_out + p * C + grp * GC);
#pragma unroll
                        for (int k = 0; k < GC / 4; k++) {
                            const float4 gv = __ldg(go + k), hv = __ldg(ho + k);
                            h[4 * k] = hv.x > 0.0f ? gv.x : 0.0f;
                            h[4 * k + 1] = hv.y > 0.0f ? gv.y : 0.0f;
                            h[4 * k + 2] = hv.z > 0.0f ? gv.z : 0.0f;
                            h[4 * k + 3] = hv.w > 0.0f ? gv.w : 0.0f;
                        }
                    } else {
#pragma unroll
                        for (int o = 0; o < GC; o++) {
                            const int c = grp * GC + o;
                            h[o] = sh.b1[c] + sh.w1[2 * c] * xn[t][0] + sh.w1[2 * c + 1] * xn[t][1];
                        }
                        if (a.acts) store_acts(a.acts + p * C + grp * GC, h);
                    }
                    store_chunk(sh, grp, (row + 3) * WP + lane + 3, h);
                }
                if (!BWD) wrote(t);
            }
            if (BWD)                                 // after all the rows, so that their loads are in flight together
                for (int t = 0; t < MT; t++) wrote(t);
        };
        int lay = 0, tile = 0, outs = 0;             // layers, tiles and last-layer tiles so far
        bool run = true;
        if (blockIdx.x < a.n) {
            fetch(blockIdx.x);
            fill(blockIdx.x);
        }
        for (int img = blockIdx.x; img < a.n && run; img += gridDim.x) {
            for (int l = 0; l < NL && run; l++, lay++) {
                const bool last = l == NL - 1;
                float keep[GC];                      // the tile before's outputs, not yet in the planes
#pragma unroll 1
                for (int t = 0; t < MT; t++, tile++) {
                    if (last && t == MT - 2 && img + (int)gridDim.x < a.n) fetch(img + gridDim.x);
                    if (!landed(&sh.accfull[t], lay)) { run = false; break; }
                    tc::fence_after();
                    float h[GC];
                    shift_sum(tl + (uint32_t)((tile & 1) * 256), h);
                    const int row = 4 * t + lq;
                    const bool mine = row < S && lane < S;
                    const long p = (long)img * NPX + row * S + lane;
                    if (!BWD) {
#pragma unroll
                        for (int o = 0; o < GC; o++) h[o] = fmaxf(h[o] + sh.bc[l][grp * GC + o], 0.0f);
                    }
                    if (!BWD && last) {              // the output's parts, summed by group 0 before it gives the buffer back
                        float s = 0.0f;
#pragma unroll
                        for (int o = 0; o < GC; o++) s = fmaf(sh.w6[grp * GC + o], h[o], s);
                        float (&part)[NG][128] = sh.ypart[outs & 1];
                        if (grp) {
                            part[grp][lq * 32 + lane] = s;
                            __syncwarp();
                            if (lane == 0) tc::mbar_arrive(&sh.yfull[outs & 1]);
                        } else {
                            if (!landed(&sh.yfull[outs & 1], outs >> 1)) { run = false; break; }
                            s = sh.b6 + s;
#pragma unroll
                            for (int g = 1; g < NG; g++) s += part[g][lq * 32 + lane];
                            if (mine) a.y[p] = s * (1.0f / NPX);
                        }
                        outs++;
                    }
                    tc::fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&sh.accempty[tile & 1]);
                    if (!last) {                     // this tile's MMAs were the last to read the rows of the one before
                        if (t) {
                            if (4 * (t - 1) + lq < S && lane < S)
                                store_chunk(sh, grp, (4 * (t - 1) + lq + 3) * WP + lane + 3, keep);
                            wrote(t - 1);
                        }
                        if (t == MT - 1) {
                            if (mine) store_chunk(sh, grp, (row + 3) * WP + lane + 3, h);
                            wrote(t);
                        }
                    } else if (t == MT - 1 && img + (int)gridDim.x < a.n) {
                        fill(img + gridDim.x);       // the image's MMAs are done
                    }
                    if (mine) {
                        if (BWD) store_acts(a.dh_in + p * C + grp * GC, h);
                        else if (a.acts) store_acts(a.acts + (long)(l + 1) * a.lstride + p * C + grp * GC, h);
                    }
#pragma unroll
                    for (int o = 0; o < GC; o++) keep[o] = h[o];
                }
            }
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (warp == 0) tc::tmem_dealloc(tmem, TMEM_COLS);
}

template <bool BWD>
int launch_tc(const CnnTcArgs& a, int num_sms, cudaStream_t st) {
    const int smem = (int)sizeof(CnnTcShared);
    const cudaError_t e = cudaFuncSetAttribute(cnn_tc_kernel<BWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return argus_cuda_fail(e);
    cnn_tc_kernel<BWD><<<a.n < num_sms ? a.n : num_sms, NTHR, smem, st>>>(a); argus_count_launch(1);
    return argus_launch_status();
}

}  // namespace

int argus_cnn_dgrad_tc(const float* dh_out, const float* h_out, const void* wbf, void* wpack, int layer, int n,
                       float* dh_in, int num_sms, int* status, cudaStream_t st) {
    cnn_pack_dgrad_tc_kernel<<<num_sms, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(wbf),
                                                       static_cast<__nv_bfloat16*>(wpack), layer); argus_count_launch(1);
    CnnTcArgs a = {};
    a.dh_out = dh_out; a.h_out = h_out; a.dh_in = dh_in; a.wpack = static_cast<const uint8_t*>(wpack);
    a.n = n; a.status = status;
    return launch_tc<true>(a, num_sms, st);
}

// The forward outside a training step (a step rounds as cnn_train_tc.cu does).
int argus_cnn_forward_tc(const float* x, const void* wbf, void* wpack, int n, float* y, float* acts, long lstride,
                         int num_sms, int* status, cudaStream_t st) {
    static_assert(sizeof(__nv_bfloat16) == 2, "BF16 storage");
    cnn_pack_tc_kernel<<<num_sms, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(wbf),
                                                 static_cast<__nv_bfloat16*>(wpack)); argus_count_launch(1);
    CnnTcArgs a = {};
    a.x = x; a.w = static_cast<const __nv_bfloat16*>(wbf); a.y = y; a.acts = acts; a.lstride = lstride;
    a.wpack = static_cast<const uint8_t*>(wpack); a.n = n; a.status = status;
    return launch_tc<false>(a, num_sms, st);
}

size_t argus_cnn_tc_pack_bytes() { return (size_t)4 * KS * KYB; }
