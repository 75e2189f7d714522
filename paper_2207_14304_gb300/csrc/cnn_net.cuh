// What the learned kernel's translation units share: the network's shape, the layout of its
// parameter vector and, for the two tensor-core forwards (cnn_tc.cu, cnn_train_tc.cu),
// their bounded waits and the BF16 hi/lo split of eight channels.
#pragma once

#include "argus_internal.cuh"
#include "split16.cuh"
#include "tc_ptx.cuh"

namespace cnn_net {

constexpr int S = 21, NPX = S * S, C = 32, KS = 7, NTAP = KS * KS;

// parameter offsets: W1 [32][2], b1, four layers of W [7][7][32][32] and b, W6, b6
constexpr long OFF_W1 = 0, OFF_B1 = 64;
__host__ __device__ constexpr long off_w(int l) { return 96 + (long)l * (49 * 1024 + 32); }
__host__ __device__ constexpr long off_b(int l) { return off_w(l) + 49 * 1024; }
constexpr long OFF_W6 = off_w(4), OFF_B6 = OFF_W6 + 32, NPARAM = OFF_B6 + 1;

constexpr long long WAIT_LIMIT = 2000000000LL;   // ~1 s of SM clock

// One try first (the common case), then a bounded wait that also gives up once
// another role has aborted.  Shared has an int `abort`.
template <typename Shared>
__device__ __forceinline__ bool wait_or_abort(Shared& sh, uint64_t* bar, uint32_t parity, int* status) {
    if (tc::mbar_try_wait(bar, parity)) return true;
    if (*(volatile int*)&sh.abort) return false;
    if (!tc::mbar_wait_bounded(bar, parity, WAIT_LIMIT)) {
        sh.abort = 1;
        argus_latch(status, ARGUS_ERR_TIMEOUT);
        return false;
    }
    return true;
}

// Eight channels as BF16 hi and lo parts (v = hi + lo + e, |e| <= 2^-17 |v|).
__device__ __forceinline__ void split_chunk(const float* h, uint8_t* dst_hi, uint8_t* dst_lo) {
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const float v0 = h[2 * k], v1 = h[2 * k + 1];
        hi[k] = bf16x2_rn(v0, v1);
        lo[k] = bf16x2_rn(v0 - __uint_as_float(hi[k] << 16), v1 - __uint_as_float(hi[k] & 0xffff0000u));
    }
    *reinterpret_cast<uint4*>(dst_hi) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst_lo) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
}

template <int N> __device__ __forceinline__ void store_acts(float* dst, const float (&h)[N]) {
#pragma unroll
    for (int k = 0; k < N / 4; k++)
        reinterpret_cast<float4*>(dst)[k] = make_float4(h[4 * k], h[4 * k + 1], h[4 * k + 2], h[4 * k + 3]);
}

}  // namespace cnn_net
