// Device helpers of the lean convolution epilogues (INT8 codes, no further
// option): scaling, rounding and the per-warp TMA store of the codes.
#pragma once

#include "hatq_internal.h"
#include "hatq_tc.h"

namespace hatq {
namespace tc {

// 4 int8 codes (one 32-bit word) -> 2 fp16x2 words, exactly: with u = b + 128
// in [0, 255], the fp16 bit pattern 0x6400 | u is 1024 + u, and subtracting
// 1152 leaves b (every step is exact in fp16).
__device__ __forceinline__ void i8x4_to_f16x4(uint32_t w, uint32_t &lo, uint32_t &hi) {
    uint32_t u = w ^ 0x80808080u, a, b;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(a) : "r"(u), "r"(0x64646464u), "r"(0x4140u));
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(b) : "r"(u), "r"(0x64646464u), "r"(0x4342u));
    asm("sub.f16x2 %0, %1, %2;" : "=r"(lo) : "r"(a), "r"(0x64806480u));
    asm("sub.f16x2 %0, %1, %2;" : "=r"(hi) : "r"(b), "r"(0x64806480u));
}

// t = M a + M b of G columns from tile column col: tensor memory, then 64-bit
// multiply-adds with the bias products staged in shared memory.
template <int G>
__device__ __forceinline__ void lean_scale(const uint32_t (&r)[G], const long long *mb, const int *mult, long long *t) {
#pragma unroll
    for (int i = 0; i < G; i += 4) {
        const int4 m = *reinterpret_cast<const int4 *>(mult + i);
        const longlong2 b0 = *reinterpret_cast<const longlong2 *>(mb + i);
        const longlong2 b1 = *reinterpret_cast<const longlong2 *>(mb + i + 2);
        t[i] = (long long)m.x * __float2int_rn(__uint_as_float(r[i])) + b0.x;
        t[i + 1] = (long long)m.y * __float2int_rn(__uint_as_float(r[i + 1])) + b0.y;
        t[i + 2] = (long long)m.z * __float2int_rn(__uint_as_float(r[i + 2])) + b1.x;
        t[i + 3] = (long long)m.w * __float2int_rn(__uint_as_float(r[i + 3])) + b1.y;
    }
}

// Codes of G columns as words of four. For a shift n >= 33 the half 2^(n-1) has
// a zero low word, so round half up is (hi + half_hi) >> (n - 32) on the high
// word alone, and half to even differs only for values whose low word is zero:
// without one in the group (the usual case) that is the rounding.
template <int G>
__device__ __forceinline__ void lean_codes(int shift, const long long (&t)[G], uint32_t (&w)[G / 4]) {
    if (shift >= 32) {
        uint32_t mn = 0xFFFFFFFFu;
#pragma unroll
        for (int i = 0; i < G; i += 2) mn = min(mn, min((uint32_t)t[i], (uint32_t)t[i + 1]));
        const int sh = shift - 32;
        if (sh > 0 && mn != 0u) {
            const int half = 1 << (sh - 1);
#pragma unroll
            for (int i = 0; i < G / 4; ++i) {
                int q[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    q[k] = max(((int)((unsigned long long)t[4 * i + k] >> 32) + half) >> sh, -127);
                w[i] = pack4_sat(q[0], q[1], q[2], q[3]);
            }
            return;
        }
        const long long kadd = (1LL << (shift - 1)) - 1;
#pragma unroll
        for (int i = 0; i < G / 4; ++i)
            w[i] = pack4_sat(requant8_lo(t[4 * i], kadd, sh), requant8_lo(t[4 * i + 1], kadd, sh),
                             requant8_lo(t[4 * i + 2], kadd, sh), requant8_lo(t[4 * i + 3], kadd, sh));
        return;
    }
#pragma unroll
    for (int i = 0; i < G / 4; ++i)
        w[i] = pack4(requant8(t[4 * i], shift), requant8(t[4 * i + 1], shift), requant8(t[4 * i + 2], shift),
                     requant8(t[4 * i + 3], shift));
}

// One warp's staging: two buffers of 32 rows of 64 bytes.
constexpr int kWarpStage = 4096;

// Codes of this lane's row (G = 64: 64 bytes, 64-byte swizzle; G = 32: 32
// bytes, 32-byte swizzle) into a staging buffer, then one TMA store of the
// warp's 32 rows. The buffer's previous store was the second last.
template <int G>
__device__ __forceinline__ void lean_store(uint8_t *buf, const uint32_t (&w)[G / 4], const CUtensorMap *tmY, int lane,
                                           bool inside, int ch, int ox, int oy, int img) {
    if (lane == 0) bulk_wait_read<1>();
    __syncwarp();
    const int sw = G == 64 ? (lane >> 1) & 3 : (lane >> 2) & 1;
#pragma unroll
    for (int q = 0; q < G / 16; ++q)
        *reinterpret_cast<uint4 *>(buf + lane * G + ((q ^ sw) << 4)) = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
    fence_async_shared();
    __syncwarp();
    if (lane == 0) {
        if (inside) tma_store_4d(smem_addr(buf), tmY, ch, ox, oy, img);
        bulk_commit();
    }
}

// ------------------------------------------------------------------ transitions
//
// Code size: 64 values per thread with each transform written out are 46 KB of
// straight-line code. Beyond about 32 KB the instruction cache misses: a warp
// then issues every 3.1 cycles instead of every 1.1 (measured on the 64-point
// transform alone), and the short loops of the other roles are evicted all the
// time. So both transforms of a transition are one copy of code in a loop of two
// passes, and loops over groups stay rolled.

// H~_out, phi, H~_next of G columns held by one thread.
template <int G>
__device__ __forceinline__ void whole_transition(long long (&t)[G], int hb_out, int hb_next, int act) {
    if (hb_out) fwht_stages<G>(t, hb_out);
    if (act) {
#pragma unroll
        for (int i = 0; i < G; ++i) t[i] = relu_mad(t[i]);
    }
    if (hb_next) fwht_stages<G>(t, hb_next);
}

// Groups shared by the two warps of a quadrant, one of each epilogue warpgroup: a
// thread finishes H = G / 2 of a row's columns, and the halves meet in the group's
// top butterfly: the lower half keeps the sums, the upper half the differences
// (lower - upper). Eight values per thread and round through the warps' staging, one
// barrier of the pair per round: rounds alternate between the two 2 KB halves, and a
// half is written again only after the next round's barrier, which the partner
// reaches after reading it. Every warp runs the barriers, also after an abort.
template <int H>
__device__ __forceinline__ void exchange_top(long long (&p)[H], uint8_t *mine_b, const uint8_t *theirs_b, int wg, int quad,
                                             int lane) {
#pragma unroll
    for (int rd = 0; rd < H / 8; ++rd) {
        int4 *mine = reinterpret_cast<int4 *>(mine_b + (rd & 1) * (kWarpStage / 2)) + lane;
        const int4 *theirs = reinterpret_cast<const int4 *>(theirs_b + (rd & 1) * (kWarpStage / 2)) + lane;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long u0 = p[8 * rd + 2 * k], u1 = p[8 * rd + 2 * k + 1];
            mine[k * 32] = make_int4((int)u0, (int)(u0 >> 32), (int)u1, (int)(u1 >> 32));
        }
        asm volatile("bar.sync %0, 64;" ::"r"(4 + quad) : "memory");
        if (wg) {
#pragma unroll
            for (int k = 0; k < 8; ++k) p[8 * rd + k] = -p[8 * rd + k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int4 v = theirs[k * 32];
            p[8 * rd + 2 * k] += (long long)(((unsigned long long)(uint32_t)v.y << 32) | (uint32_t)v.x);
            p[8 * rd + 2 * k + 1] += (long long)(((unsigned long long)(uint32_t)v.w << 32) | (uint32_t)v.z);
        }
    }
}

// From t = M a + M b to the stored codes of this warp's half group (channels ch ..
// ch + H - 1 of the box at (ox, oy) of image img). The codes take the staging half
// that the exchange's last round did not use.
template <int G>
__device__ __forceinline__ void split_finish(long long (&t)[G / 2], int shift, int hb_out, int hb_next, int act, uint8_t *wstage,
                                             const uint8_t *theirs, int wg, int quad, int lane, const CUtensorMap *tmY,
                                             bool inside, int ch, int ox, int oy, int img) {
    constexpr int H = G / 2;
    if (lane == 0) bulk_wait_read<0>();                  // the previous group's store has left the staging
    __syncwarp();
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        const int hb = pass ? hb_next : hb_out;
        if (hb == G) {
            if (pass && hb_out == G)                     // the partner has read the first exchange's last round
                asm volatile("bar.sync %0, 64;" ::"r"(4 + quad) : "memory");
            exchange_top<H>(t, wstage, theirs, wg, quad, lane);
        }
        if (hb) fwht_stages<H>(t, min(hb, H));
        if (!pass && act) {
#pragma unroll
            for (int i = 0; i < H; ++i) t[i] = relu_mad(t[i]);
        }
    }
    uint32_t w[H / 4];
    lean_codes<H>(shift, t, w);
    lean_store<H>(wstage, w, tmY, lane, inside, ch, ox, oy, img);
}

}  // namespace tc
}  // namespace hatq
