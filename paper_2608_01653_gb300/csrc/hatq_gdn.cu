// The GDN / IGDN transition of the supplementary's general nonlinearities
// (Eqs. supp_general_activation, supp_general_input_scale,
// supp_general_input_transition) for channel-coupled activations, on the
// 5th-generation tensor cores.
//
// Input: the integer preactivation z (Eq. supp_general_preactivation), one
// row of c INT8 codes per pixel, as a plain layer with output scale s_z emits
// it. Per pixel:
//   D_i = B_i + sum_j G_ij z_j^2                        (the normalization pool)
//   |u_i| = largest k <= 127 with (2k - 1)^2 D_i 2^t <= 4 P z_i^2     (GDN)
//           largest k <= 127 with (2k - 1)^2 2^t <= 4 P z_i^2 D_i     (IGDN)
//   u_i with the sign of z_i, i.e. round(R |z_i| / sqrt(D_i)) (IGDN: times
//   sqrt(D_i)) with ties away from zero and R^2 = P / 2^t;
//   x = clamp(round(H~_next (M_in u) / 2^n_in), -127, 127).
//
// The pool is a dense contraction over channels: D = Z2 G^T for a tile of
// 128 pixels, Z2 the squared codes. z^2 <= 16129 is split into two limbs
// z^2 = 128 h + l with h = round(z^2 / 128) <= 126 and |l| <= 64; G <= 511 and the
// limbs are exact in fp16, every product is <= 511 * 126 and a sum over c <= 256
// channels stays below 2^24, so the two fp32 accumulators in tensor memory are
// exact. The limbs come straight from fp16 arithmetic on y = z / 16, two values per
// instruction: t = fma(y, y, 768) rounds z^2 / 256 to a multiple of 1/2, so
// t - 768 = h / 2 and fma(y, y, -h / 2) = l / 256, both exact, and
// D = 256 (D_h + D_l) + B with the accumulators of these scaled limbs.
//
// Persistent kernel, one CTA per SM, 640 threads in five warpgroups:
//   warp 0       TMA: G once (resident, 128-byte swizzle), the z tiles (c / 64 boxes
//                of 64 x 128 bytes, 64-byte swizzle, 2-4 tiles ahead)
//   warp 1       TMEM allocation; MMAs: per tile c / 64 passes of 64 output channels,
//                both limbs by c / 16 K-steps into accumulator buffer unit & 1
//   warps 4-7    limbs of z^2 of the tile's 128 rows into TMEM (the A operand)
//   warps 8-19   three warpgroups take the units (tile, pass) in turn; a thread
//                finishes the 64 channels of its pixel row by itself: code estimate
//                and exact corrections, Sylvester block in registers, a table of
//                clamp(round(M_in v / 2^n_in)) over |v| <= 127 hb (built once per
//                CTA), one TMA store of 64 bytes x 32 rows per warp
// No warp waits for another but through the barriers of tiles, limbs and accumulators;
// every wait is bounded.
// Bound: 32 instructions per value, issued at about 48 % of the rate (waits on tensor and shared
// memory take the rest; the memory traffic alone would take 117 us for 4 x 540 x 960 x 192). That size takes 704 us; with quarters of a pixel row in different
// warps, CTA-wide barriers between the phases and 59 instructions per value it took 1561.
// Straight code beyond the instruction cache is what costs next: with the exact
// corrections unrolled per value it took 2424 us, as one rolled loop over the marked
// channels 951, with the table's address and the scale folded in 762, and without loop
// exits between the butterfly stages (a move per value each) 704.
#include <cuda_fp16.h>

#include "hatq_internal.h"
#include "hatq_launch.h"
#include "hatq_tc.h"

namespace hatq {
namespace {

using namespace tc;

constexpr int kGdnThreads = 640;
constexpr int kPoolGroups = 3;                  // warpgroups that finish units
constexpr int kMaxZ = 4;                        // z tile buffers at most

// |u| for one channel, exactly: the largest k <= 127 with (2k - 1)^2 den <= num
// (GDN: den = D 2^t, num = 4 P a^2; IGDN: den = 2^t, num = 4 P a^2 D), i.e.
// round(X) with ties up for X = a sqrt(P / (2^t D)) (IGDN: a sqrt(P D / 2^t)),
// searched from the estimate k0 (the loops make it exact whatever k0 is).
__device__ __forceinline__ int gdn_code_exact(uint32_t ab, uint32_t D, int k0, const GdnArgs &a) {
    unsigned long long num = 4ull * a.P * (unsigned long long)(ab * ab);
    unsigned long long den;
    if (a.inverse) {
        num *= D;
        den = 1ull << a.t;
    } else {
        den = (unsigned long long)D << a.t;
    }
    auto cond = [&](int kk) {
        const unsigned long long o = (unsigned long long)(2 * kk - 1);
        return o * o * den <= num;
    };
    int k = k0 < 0 ? 0 : (k0 > 127 ? 127 : k0);
    while (k < 127 && cond(k + 1)) ++k;
    while (k > 0 && !cond(k)) --k;
    return k;
}

// Two code words (8 codes) as y = z / 16 in fp16 pairs, exactly: the fp16 pattern
// 0x6400 | (z + 128) is 1152 + z, times 2^-4 minus 72.
__device__ __forceinline__ void y_pairs(uint32_t w, uint32_t &lo, uint32_t &hi) {
    const uint32_t u = w ^ 0x80808080u, a = __byte_perm(u, 0x64646464u, 0x4140), b = __byte_perm(u, 0x64646464u, 0x4342);
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(lo) : "r"(a), "r"(0x2C002C00u), "r"(0xD480D480u));
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(hi) : "r"(b), "r"(0x2C002C00u), "r"(0xD480D480u));
}
// The scaled limbs of two codes: h / 2 and l / 256.
__device__ __forceinline__ void limb_pair(uint32_t y, uint32_t &h, uint32_t &l) {
    uint32_t t, nh;
    asm("fma.rn.f16x2 %0, %1, %1, %2;" : "=r"(t) : "r"(y), "r"(0x62006200u));           // + 768
    asm("sub.f16x2 %0, %1, %2;" : "=r"(h) : "r"(t), "r"(0x62006200u));
    asm("neg.f16x2 %0, %1;" : "=r"(nh) : "r"(h));
    asm("fma.rn.f16x2 %0, %1, %1, %2;" : "=r"(l) : "r"(y), "r"(nh));
}

__device__ __forceinline__ void umma_f16_ts_if(uint32_t pr, uint32_t d_tmem, uint32_t a_tmem, uint32_t blo, uint32_t bhi,
                                               uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .b64 db;\n mov.b64 db, {%2, %3};\n setp.ne.b32 p, %5, 0;\n setp.ne.b32 q, %6, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc), "r"(pr)
        : "memory");
}
__device__ __forceinline__ int lds_u8(uint32_t addr) {
    uint32_t r;
    asm("ld.shared.u8 %0, [%1];" : "=r"(r) : "r"(addr));
    return (int)r;
}
__device__ __forceinline__ void tma_store_2d(uint32_t src, const CUtensorMap *tm, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%1, {%2, %3}], [%0];" ::"r"(src), "l"(tm), "r"(c0),
                 "r"(c1)
                 : "memory");
}

// The float estimate of one channel, X = z rsqrt(d) with d = D 2^t / P (IGDN: z sqrt(d),
// d = D P / 2^t), clamped to [-127, 127]; d = k256 (D_h + D_l) + B', the factor in k256 and B'.
// D_h and D_l are exact, 256 D_h <= 2 D and 256 |D_l| <= D, so d's relative error is at most
// 5 x 2^-24 (k256 3, two fmas 2), half of that after the square root; with rsqrt.approx
// (2^-22.9) and at most two products X is off by less than 127.5 x 4.0e-7 < 2^-14: it decides
// every code whose |X| lies more than 2^-14 from a half-integer.
constexpr uint32_t kCodeBias = 0x4B400000u;           // bits of 1.5 2^23
constexpr float kSure = 0.5f - 0.00006103515625f;
template <bool INV>
__device__ __forceinline__ float gdn_estimate(float zf, uint32_t dh, uint32_t dl, float bf, float k256) {
    const float df = fmaf(k256, __uint_as_float(dh), fmaf(k256, __uint_as_float(dl), bf));
    float r, y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(df));
    const float x = INV ? zf * (df * r) : zf * r;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(y) : "f"(x), "f"(127.0f));   // sign(x) min(|x|, 127)
    return y;
}

template <bool INV>
__global__ void __launch_bounds__(kGdnThreads, 1)
    gdn_kernel(const __grid_constant__ CUtensorMap tmZ, const __grid_constant__ CUtensorMap tmG,
               const __grid_constant__ CUtensorMap tmY, const __grid_constant__ GdnArgs a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int c = a.c, np = c / 64;
    const int zbytes = 128 * c;
    uint8_t *z_s = smem + a.z_off;                         // nz x [c / 64][128 rows][64 B], 64-byte swizzle
    float *bf_s = reinterpret_cast<float *>(smem + a.b_off);
    const uint32_t bar0 = smem_addr(smem + a.bar_off);
    // barriers: z_full[4], z_empty[4], acc_full[3] (one per pool group: a group sees every phase of its
    // own), acc_empty[2] (one per accumulator buffer), g, a_full, a_empty
    auto z_full = [&](int b) { return bar0 + 8u * b; };
    auto z_empty = [&](int b) { return bar0 + 8u * (4 + b); };
    auto acc_full = [&](int b) { return bar0 + 8u * (8 + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (11 + b); };
    const uint32_t g_bar = bar0 + 104u, a_full = bar0 + 112u, a_empty = bar0 + 120u;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem + a.bar_off + 128);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + a.bar_off + 132);

    __shared__ int s_skip;
    if (threadIdx.x == 0) s_skip = *reinterpret_cast<volatile int *>(a.err);
    __syncthreads();
    if (s_skip != 0) return;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int quad = warp & 3, m = quad * 32 + lane;       // TMEM lane quadrant, pixel row of the tile
    const int my_tiles = a.num_tiles > (int)blockIdx.x ? (a.num_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    if (threadIdx.x == 0) {
        for (int b = 0; b < kMaxZ; ++b) {
            mbar_init(z_full(b), 1);
            mbar_init(z_empty(b), 4 + 4 * np);             // limb warps and each unit's pool warps
        }
        for (int b = 0; b < kPoolGroups; ++b) mbar_init(acc_full(b), 1);
        for (int b = 0; b < 2; ++b) mbar_init(acc_empty(b), 4);
        mbar_init(g_bar, 1);
        mbar_init(a_full, 4);
        mbar_init(a_empty, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc512<false>(smem_addr(tmem_holder));
    for (int i = threadIdx.x; i < c; i += kGdnThreads) bf_s[i] = (float)(a.b_pool[i] * a.factor);
    // x = clamp(round(M_in v / 2^n_in)) for every v = H~ u, |v| <= 127 hb; lut_s[v]
    const int vmax = 127 * (a.hb_next > 1 ? a.hb_next : 1);
    int8_t *lut_s = reinterpret_cast<int8_t *>(smem + a.lut_off) + vmax;
    const uint32_t lut = smem_addr(lut_s);
    for (int v = -vmax + (int)threadIdx.x; v <= vmax; v += kGdnThreads)
        lut_s[v] = (int8_t)requant8_any(a.mult_in * (long long)v, a.shift_in);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_holder;
    auto warp_arrive = [&](uint32_t bar) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };

    // TMEM: the limbs at columns [0, c / 2) and [c / 2, c); accumulator buffer b at c + 128 b holds
    // 64 columns of each limb's sums. Registers (launch 640 x 96): 40 + 56 + 3 x 128 = 480 = 5 x 96.
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;" ::: "memory");
        const uint32_t lead = elect_one() ? 1u : 0u;
        if (warp == 0) {
            if (my_tiles > 0) {
                mbar_expect_tx_if(lead, g_bar, (uint32_t)(c * c * 2));
                for (int kb = 0; kb < np; ++kb) tma_load_2d_if(lead, smem_addr(smem + kb * c * 128), &tmG, g_bar, 64 * kb, 0);
            }
            int b = 0;
            uint32_t ph = 1;
            for (int j = 0; j < my_tiles; ++j) {
                const int tile = (int)blockIdx.x + j * (int)gridDim.x;
                mbar_wait_issue<false>(z_empty(b), ph, abort_flag, a.err, tmem, false);
                mbar_expect_tx_if(lead, z_full(b), (uint32_t)zbytes);
                for (int cb = 0; cb < np; ++cb)
                    tma_load_2d_if(lead, smem_addr(z_s + (size_t)b * zbytes + cb * 8192), &tmZ, z_full(b), 64 * cb, 128 * tile);
                if (++b == a.nz) { b = 0; ph ^= 1u; }
            }
        } else if (warp == 1 && my_tiles > 0) {
            const uint32_t idesc = idesc_f16(64), bhi = (1024u >> 4) | (1u << 14) | (2u << 29);
            const uint32_t blo0 = ((smem_addr(smem) >> 4) & 0x3FFFu) | (1u << 16);
            const uint32_t kb_step = (uint32_t)(c * 128) >> 4, p_step = (64u * 128u) >> 4;
            mbar_wait_issue<false>(g_bar, 0, abort_flag, a.err, tmem, true);
            int u = 0, grp = 0;
            for (int j = 0; j < my_tiles; ++j) {
                mbar_wait_issue<false>(a_full, (uint32_t)(j & 1), abort_flag, a.err, tmem, true);
                for (int p = 0; p < np; ++p, ++u) {
                    const int b = u & 1;
                    if (u >= 2) mbar_wait_issue<false>(acc_empty(b), ((u >> 1) - 1) & 1, abort_flag, a.err, tmem, true);
                    tc_fence_after();
                    for (int limb = 0; limb < 2; ++limb) {
                        const uint32_t d = (uint32_t)(c + 128 * b + 64 * limb);
                        uint32_t at = (uint32_t)(limb * (c / 2)), bl = blo0 + (uint32_t)p * p_step, acc = 0;
                        for (int kb = 0; kb < np; ++kb, bl += kb_step, at += 32) {
                            umma_f16_ts_if(lead, d, at, bl, bhi, idesc, acc);
                            umma_f16_ts_if(lead, d, at + 8, bl + 2, bhi, idesc, 1u);
                            umma_f16_ts_if(lead, d, at + 16, bl + 4, bhi, idesc, 1u);
                            umma_f16_ts_if(lead, d, at + 24, bl + 6, bhi, idesc, 1u);
                            acc = 1u;
                        }
                    }
                    umma_commit_if<false>(lead, acc_full(grp));
                    grp = grp == kPoolGroups - 1 ? 0 : grp + 1;
                }
                umma_commit_if<false>(j + 1 < my_tiles ? lead : 0u, a_empty);   // (the last is not waited for)
            }
        }
    } else if (warp < 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;" ::: "memory");
        // ------------------------------------------------------ limbs
        const uint32_t t_lane = tmem + ((uint32_t)(quad * 32) << 16);
        const int sw = (m >> 1) & 3;
        int b = 0;
        uint32_t ph = 0;
        for (int j = 0; j < my_tiles; ++j) {
            bool ok = __all_sync(0xffffffffu, mbar_wait(z_full(b), ph, abort_flag, a.err));
            if (ok && j > 0) ok = __all_sync(0xffffffffu, mbar_wait(a_empty, (uint32_t)((j - 1) & 1), abort_flag, a.err));
            if (!ok) break;
            tc_fence_after();
            const uint8_t *zt = z_s + (size_t)b * zbytes + m * 64;
#pragma unroll 1
            for (int cb = 0; cb < np; ++cb) {
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    uint32_t h[16], l[16];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(zt + cb * 8192 + (((2 * hf + q) ^ sw) << 4));
                        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            uint32_t y0, y1;
                            y_pairs(w[i], y0, y1);
                            limb_pair(y0, h[8 * q + 2 * i], l[8 * q + 2 * i]);
                            limb_pair(y1, h[8 * q + 2 * i + 1], l[8 * q + 2 * i + 1]);
                        }
                    }
                    tmem_st16(t_lane + (uint32_t)(32 * cb + 16 * hf), h);
                    tmem_st16(t_lane + (uint32_t)(c / 2 + 32 * cb + 16 * hf), l);
                }
            }
            tmem_wait_st();
            tc_fence_before();
            warp_arrive(a_full);
            if (lane == 0) mbar_arrive(z_empty(b));
            if (++b == a.nz) { b = 0; ph ^= 1u; }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 128;" ::: "memory");
        // ------------------------------------------------------ pool, codes, transition
        const uint32_t t_lane = tmem + ((uint32_t)(quad * 32) << 16);
        const int sw = (m >> 1) & 3;
        uint8_t *stage = smem + a.u_off + (warp - 8) * 2048;       // 32 rows x 64 bytes, 64-byte swizzle
        const int total = my_tiles * np;
        int p = (warp - 8) >> 2, j = 0;                            // this unit's pass and tile
        const uint32_t full = acc_full((warp - 8) >> 2);
        int zb = 0;
        uint32_t zph = 0, fph = 0;
        for (int u = (warp - 8) >> 2; u < total; u += kPoolGroups, p += kPoolGroups) {
            while (p >= np) {
                p -= np;
                ++j;
                if (++zb == a.nz) { zb = 0; zph ^= 1u; }
            }
            const int db = u & 1;
            // (the accumulators first: with them ready the tile's barrier is in this tile's phase)
            bool ok = __all_sync(0xffffffffu, mbar_wait(full, fph, abort_flag, a.err));
            if (ok) ok = __all_sync(0xffffffffu, mbar_wait(z_full(zb), zph, abort_flag, a.err));
            if (!ok) break;
            fph ^= 1u;
            tc_fence_after();
            const uint8_t *zt = z_s + (size_t)zb * zbytes + p * 8192 + m * 64;
            const uint32_t t_acc = t_lane + (uint32_t)(c + 128 * db);
            // Codes as the bits of 1.5 2^23 + u; the bias leaves in the first butterflies. An estimate
            // too close to a rounding boundary sets its bit of `unsure`.
            uint32_t v[64];
            uint32_t unsure[2] = {0u, 0u};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t dh[16], dl[16];
                tmem_ld16(t_acc + 16 * q, dh);
                tmem_ld16(t_acc + 64 + 16 * q, dl);
                const uint4 zv = *reinterpret_cast<const uint4 *>(zt + ((q ^ sw) << 4));
                const float4 *bf = reinterpret_cast<const float4 *>(bf_s + 64 * p + 16 * q);
                const uint32_t zw[4] = {zv.x ^ 0x80808080u, zv.y ^ 0x80808080u, zv.z ^ 0x80808080u, zv.w ^ 0x80808080u};
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 b4 = bf[i];
                    const float b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int e = 16 * q + 4 * i + k;
                        const float zf = __uint_as_float(__byte_perm(zw[i], 0x4B000000u, 0x7650 | k)) - 8388736.0f;
                        const float x = gdn_estimate<INV>(zf, dh[4 * i + k], dl[4 * i + k], b[k], a.k256);
                        const float t = x + 12582912.0f;
                        if (fabsf(x - (t - 12582912.0f)) >= kSure) unsure[e >> 5] |= 1u << (e & 31);
                        v[e] = __float_as_uint(t);
                    }
                }
            }
            uint32_t todo[2] = {__reduce_or_sync(0xffffffffu, unsure[0]), __reduce_or_sync(0xffffffffu, unsure[1])};
            while (todo[0] | todo[1]) {                            // about every second unit of a warp: one channel
                const int e = todo[0] ? __ffs((int)todo[0]) - 1 : 31 + __ffs((int)todo[1]);
                const bool mine = ((e < 32 ? unsure[0] : unsure[1]) >> (e & 31)) & 1u;
                if (e < 32) todo[0] &= todo[0] - 1u;
                else todo[1] &= todo[1] - 1u;
                uint32_t dh, dl;
                tmem_ld1(t_acc + (uint32_t)e, dh);
                tmem_ld1(t_acc + 64 + (uint32_t)e, dl);
                tmem_wait_ld();
                uint32_t k = 0;
                if (mine) {
                    const int zi = reinterpret_cast<const int8_t *>(zt)[(((e >> 4) ^ sw) << 4) + (e & 15)];
                    const float x = gdn_estimate<INV>((float)zi, dh, dl, bf_s[64 * p + e], a.k256);
                    const uint32_t D = (uint32_t)__float2int_rn(__uint_as_float(dh) * 2.0f) * 128u +
                                       (uint32_t)__float2int_rn(__uint_as_float(dl) * 256.0f) + (uint32_t)a.b_pool[64 * p + e];
                    const int u8 = gdn_code_exact((uint32_t)abs(zi), D, (int)(fabsf(x) + 0.5f), a);
                    k = (uint32_t)(zi < 0 ? -u8 : u8) + kCodeBias;
                }
                const uint32_t bit = mine ? 1u << (e & 31) : 0u, b0 = e < 32 ? bit : 0u, b1 = e < 32 ? 0u : bit;
#pragma unroll
                for (int i = 0; i < 64; ++i)                       // (bits of a mask: v stays in registers)
                    if ((i < 32 ? b0 : b1) & (1u << (i & 31))) v[i] = k;
            }
            tc_fence_before();                                     // every read of the buffers is done
            warp_arrive(acc_empty(db));
            if (lane == 0) mbar_arrive(z_empty(zb));
            // v - bias of the first butterflies, exact (|H~ u| <= 127 hb), plus the table's address: added to
            // a full block's first value it reaches every sum, as the block's first column is all ones
            auto first = [&]() {
#pragma unroll
                for (int i = 0; i < 64; i += 2) {
                    const uint32_t s0 = v[i], s1 = v[i + 1];
                    v[i] = s0 + s1 - 2u * kCodeBias;
                    v[i + 1] = s0 - s1;
                }
            };
            auto butterflies = [&](int m2) {
#pragma unroll
                for (int i = 0; i < 64; ++i)
                    if (!(i & m2)) {
                        const uint32_t s0 = v[i], s1 = v[i | m2];
                        v[i] = s0 + s1;
                        v[i | m2] = s0 - s1;
                    }
            };
            if (a.hb_next == 64) {                                 // straight through: a stage that may be the last costs moves
                v[0] += lut;
                first();
#pragma unroll
                for (int m2 = 2; m2 < 64; m2 <<= 1) butterflies(m2);
            } else {
                if (a.hb_next > 1) {
                    first();
#pragma unroll
                    for (int m2 = 2; m2 < 32; m2 <<= 1) {
                        if (m2 >= a.hb_next) break;
                        butterflies(m2);
                    }
                }
                const uint32_t base = lut - (a.hb_next > 1 ? 0u : kCodeBias);
#pragma unroll
                for (int i = 0; i < 64; ++i) v[i] += base;
            }
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    w[i] = pack4(lds_u8(v[16 * q + 4 * i]), lds_u8(v[16 * q + 4 * i + 1]), lds_u8(v[16 * q + 4 * i + 2]),
                                 lds_u8(v[16 * q + 4 * i + 3]));
                *reinterpret_cast<uint4 *>(stage + lane * 64 + ((q ^ sw) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
            fence_async_shared();
            __syncwarp();
            const long long pix = (long long)((int)blockIdx.x + j * (int)gridDim.x) * 128 + quad * 32;
            if (lane == 0 && pix < a.pixels) {
                tma_store_2d(smem_addr(stage), &tmY, 64 * p, (int)pix);
                bulk_commit();
            }
        }
        if (lane == 0) bulk_wait_all();
    }
    tc_fence_before();
    group_sync<false>();
    tc_fence_after();
    if (warp == 1) tmem_dealloc512<false>(tmem);
}

}  // namespace

// One CTA per SM, at most one per tile.
cudaError_t launch_gdn(const CUtensorMap &tmZ, const CUtensorMap &tmG, const CUtensorMap &tmY, const GdnArgs &a, int smem_bytes,
                       cudaStream_t s) {
    auto kern = a.inverse ? gdn_kernel<true> : gdn_kernel<false>;
    static SmemOptIn opt_in[2];
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = current_device(&dev)) != cudaSuccess ||
        (e = opt_in[a.inverse ? 1 : 0].set(dev, reinterpret_cast<const void *>(kern))) != cudaSuccess ||
        (e = device_sms(dev, &sms)) != cudaSuccess)
        return e;
    const int grid = a.num_tiles < sms ? a.num_tiles : sms;
    kern<<<grid, kGdnThreads, smem_bytes, s>>>(tmZ, tmG, tmY, a);
    return cudaGetLastError();
}

}  // namespace hatq
