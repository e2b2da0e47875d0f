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
// Code size: beyond about 32 KB of straight-line code the instruction cache misses: a
// warp then issues every 3.1 cycles instead of every 1.1 (measured on the 64-point
// transform alone), and the short loops of the other roles are evicted all the time.
// 64 int64 values per thread with both transforms written out are 46 KB. So groups
// that one thread holds whole take the fp32 estimate below, and shared groups run both
// transforms as one copy of code in a loop of two passes.

// Pairs of floats, one instruction for both.
__device__ __forceinline__ uint64_t f2_pack(float x, float y) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ uint64_t f2_add(uint64_t x, uint64_t y) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(x), "l"(y));
    return d;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t x, uint64_t y, uint64_t z) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(x), "l"(y), "l"(z));
    return d;
}

// Unnormalized Sylvester transform of every hb-block of G floats (pairs of neighbours).
// Whole groups (the usual case) run straight through: where a stage may be the last,
// every value has to be moved to the register that the others leave it in.
template <int G>
__device__ __forceinline__ void f2_fwht(uint64_t (&p)[G / 2], int hb) {
    const uint64_t neg = f2_pack(-1.0f, -1.0f);
    auto first = [&]() {
#pragma unroll
        for (int i = 0; i < G / 2; ++i) {
            float x, y;
            f2_unpack(p[i], x, y);
            p[i] = f2_pack(x + y, x - y);
        }
    };
    auto stage = [&](int h) {
#pragma unroll
        for (int i = 0; i < G / 2; ++i)
            if (!(i & h)) {
                const uint64_t x = p[i], y = p[i + h];
                p[i] = f2_add(x, y);
                p[i + h] = f2_fma(y, neg, x);
            }
    };
    if (hb == G) {
        first();
#pragma unroll
        for (int h = 1; h < G / 2; h <<= 1) stage(h);
    } else if (hb > 1) {
        first();
#pragma unroll
        for (int h = 1; h < G / 4; h <<= 1) {
            if (2 * h >= hb) break;
            stage(h);
        }
    }
}

// Constants of the estimate in shared memory, 16 bytes a channel: multipliers and bias
// products times 2^-n in fp32, each rounded once, then multipliers and bias codes.
__device__ __forceinline__ void stage_quick(float *s, const int32_t *mult, const int32_t *b_int, int co, int shift) {
    const float sc = __int_as_float((127 - max(shift, 0)) << 23);
    for (int c = threadIdx.x; c < co; c += blockDim.x) {
        const int m = mult[c], b = b_int[c];
        s[c] = (float)m * sc;
        s[co + c] = (float)((long long)m * b) * sc;
        reinterpret_cast<int *>(s)[2 * co + c] = m;
        reinterpret_cast<int *>(s)[3 * co + c] = b;
    }
}

// The transition's options and the factors of the estimate's error bound (quick_codes).
struct Quick {
    int hb_out, hb_next, act, shift;
    float kf, kb, kz;
};
template <int G>
__device__ __forceinline__ Quick quick_setup(int hb_out, int hb_next, int act, int shift) {
    const int h1 = hb_out > 1 ? hb_out : 1, h2 = hb_next > 1 ? hb_next : 1;
    const float u = 1.02f / 16777216.0f, g = sqrtf((float)h1 * (float)h2) * u;
    const float l1 = (float)(31 - __clz(h1)), l2 = (float)(31 - __clz(h2));
    const bool dc = act && hb_next == G;                     // the first output is the sum of phi's values
    return Quick{hb_out, hb_next, act, shift, g * (2.0f + l1 + (dc ? 0.0f : l2)), g * 2.0f, dc ? u * l2 : 0.0f};
}

// Codes of one row's G columns, a[] the exact sums: t = M a + M b, H~_out, phi, H~_next
// and round(t / 2^n), estimated in fp32 with every factor already times 2^-n. Returns
// whether each code is certain. u = 2^-24:
//   Factor, bias and multiply-add are each rounded, so a value f with bias term b is off by
//   at most 2u (|f| + |b|), the row by 2u (F + B) in norm (F, B the norms of f and b).
//   A stage of a transform of size h rounds its sums, u of their norm; the transform
//   scales a vector's norm by sqrt(h), phi never lengthens a difference, and one output
//   of the last transform is at most sqrt(h) times the norm of its input: an output is off
//   by at most sqrt(h_out h_next) u (2 (F + B) + (log2 h_out + log2 h_next) F). After a
//   ReLU the last transform's own rounding is at most u log2 h_next times the sum of its
//   inputs, which is its first output.
// A value farther than that from every half-integer has the exact value's rounding; the
// others take exact_rows (one row in a hundred of a 5x5 3 -> 192 layer with a 64-wide
// output and input transform). That layer on 8 x 2160 x 3840: 4256 us, of 6480 with 64
// int64 values per thread; with a loop exit after each butterfly stage 5811 (20
// instructions on the multiply-add pipe per value instead of 12, mostly moves), with
// both transforms written out as well 7156 (instruction cache).
template <int G>
__device__ __forceinline__ bool quick_codes(const uint32_t (&a)[G], const float *ms, const float *bs, const Quick &o, int lane,
                                            uint32_t (&w)[G / 4]) {
    uint64_t p[G / 2], n0 = 0, n1 = 0;
#pragma unroll
    for (int i = 0; i < G; i += 4) {
        const float4 m = *reinterpret_cast<const float4 *>(ms + i), b = *reinterpret_cast<const float4 *>(bs + i);
        p[i / 2] = f2_fma(f2_pack(__uint_as_float(a[i]), __uint_as_float(a[i + 1])), f2_pack(m.x, m.y), f2_pack(b.x, b.y));
        p[i / 2 + 1] = f2_fma(f2_pack(__uint_as_float(a[i + 2]), __uint_as_float(a[i + 3])), f2_pack(m.z, m.w), f2_pack(b.z, b.w));
        n0 = f2_fma(p[i / 2], p[i / 2], n0);
        n1 = f2_fma(p[i / 2 + 1], p[i / 2 + 1], n1);
    }
    float x, y, bb = bs[lane] * bs[lane];
    if (G == 64) bb = fmaf(bs[lane + 32], bs[lane + 32], bb);
#pragma unroll
    for (int d = 16; d; d >>= 1) bb += __shfl_xor_sync(0xffffffffu, bb, d);
    f2_unpack(f2_add(n0, n1), x, y);
    float sure = 0.4999998f - fmaf(o.kf, sqrtf(x + y), o.kb * sqrtf(bb));
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        f2_fwht<G>(p, pass ? o.hb_next : o.hb_out);
        if (!pass && o.act) {
#pragma unroll
            for (int i = 0; i < G / 2; ++i) {
                f2_unpack(p[i], x, y);
                p[i] = f2_pack(fmaxf(x, 0.f), fmaxf(y, 0.f));
            }
        }
    }
    f2_unpack(p[0], x, y);
    sure = fmaf(-o.kz, x, sure);
    const uint64_t bias = f2_pack(12582912.0f, 12582912.0f), back = f2_pack(-12582912.0f, -12582912.0f),
                   neg = f2_pack(-1.0f, -1.0f);
    float worst = 0.f;
#pragma unroll
    for (int i = 0; i < G / 4; ++i) {
        float t[4];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            f2_unpack(p[2 * i + k], x, y);
            asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(x) : "f"(x), "f"(127.0f));      // sign(x) min(|x|, 127)
            asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(y) : "f"(y), "f"(127.0f));
            const uint64_t v = f2_pack(x, y), r = f2_add(v, bias);
            f2_unpack(r, t[2 * k], t[2 * k + 1]);                                        // low byte: the code
            f2_unpack(f2_fma(f2_add(r, back), neg, v), x, y);                            // exact
            asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(worst) : "f"(worst), "f"(x), "f"(y));
        }
        w[i] = pack4(__float_as_int(t[0]), __float_as_int(t[1]), __float_as_int(t[2]), __float_as_int(t[3]));
    }
    return worst < sure;
}

constexpr int kWarpScratch = 512;

// round(v / 2^n) half to even, clamped to [-127, 127], in few instructions of code.
__device__ __forceinline__ int exact_code(long long v, int n) {
    if (n > 0) v = (v + ((1LL << (n - 1)) - 1) + ((v >> n) & 1)) >> n;
    return (int)(v > 127 ? 127 : (v < -127 ? -127 : v));
}

// The codes of the rows (lanes) in `rows`, exactly: the warp takes two rows at a time, half
// a warp each and C neighbouring columns per lane, in int64 with shuffles. mult / b_int:
// the group's channels in shared memory.
template <int G>
__device__ __forceinline__ void exact_rows(uint32_t rows, const uint32_t (&a)[G], const int *mult, const int *b_int,
                                           const Quick &o, uint8_t *scratch, int lane, uint32_t (&w)[G / 4]) {
    constexpr int C = G / 16;
    const int col = C * (lane & 15);
    uint8_t *half = scratch + (lane >> 4) * 256;
    while (rows) {
        const int r0 = __ffs((int)rows) - 1;
        rows &= rows - 1u;
        const int r1 = rows ? __ffs((int)rows) - 1 : r0;
        rows &= rows - 1u;
        const bool owner = lane == r0 || lane == r1;
        uint8_t *own = scratch + (lane == r0 ? 0 : 256);
        if (owner) {
#pragma unroll
            for (int i = 0; i < G; i += 4)
                *reinterpret_cast<uint4 *>(own + 4 * i) = make_uint4(a[i], a[i + 1], a[i + 2], a[i + 3]);
        }
        __syncwarp();
        long long t[C];
#pragma unroll
        for (int k = 0; k < C; ++k)
            t[k] = (long long)mult[col + k] * (__float2int_rn(reinterpret_cast<const float *>(half)[col + k]) + (long long)b_int[col + k]);
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            const int hb = pass ? o.hb_next : o.hb_out;
#pragma unroll
            for (int h = 1; h < C; h <<= 1) {
                if (h >= hb) break;
#pragma unroll
                for (int k = 0; k < C; ++k)
                    if (!(k & h)) {
                        const long long x = t[k], y = t[k + h];
                        t[k] = x + y;
                        t[k + h] = x - y;
                    }
            }
#pragma unroll 1
            for (int d = 1; d * C < hb; d <<= 1) {
                const bool upper = (lane & d) != 0;
#pragma unroll
                for (int k = 0; k < C; ++k) {
                    const long long x = __shfl_xor_sync(0xffffffffu, t[k], d);
                    t[k] = x + (upper ? -t[k] : t[k]);
                }
            }
            if (!pass && o.act) {
#pragma unroll
                for (int k = 0; k < C; ++k) t[k] = t[k] > 0 ? t[k] : 0;
            }
        }
        __syncwarp();                                        // the values have been read
#pragma unroll
        for (int k = 0; k < C; ++k) half[col + k] = (uint8_t)exact_code(t[k], o.shift);
        __syncwarp();
        if (owner) {
#pragma unroll
            for (int i = 0; i < G / 16; ++i) {
                const uint4 v = reinterpret_cast<const uint4 *>(own)[i];
                w[4 * i] = v.x;
                w[4 * i + 1] = v.y;
                w[4 * i + 2] = v.z;
                w[4 * i + 3] = v.w;
            }
        }
        __syncwarp();                                        // before the next rows' values
    }
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
