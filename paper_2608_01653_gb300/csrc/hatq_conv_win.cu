// INT8 convolution with the fused requantize / Hadamard epilogue (Eqs.
// linear_operator, integer_accumulation, integer_hadamard_transition) for
// layers with c_in % 16 == 0: the window form of conv_kernel.
//
// The tensor cores take the codes as exact fp16 values, so the INT8 operand has
// to be converted. conv_kernel converts it again for every kernel tap (25 times
// for a 5x5 layer); at about 115 warp instructions per 64-code row and tap that
// conversion, not the MMAs, bounded the large layers (307 issue slots per
// scheduler and 64-wide block against 256 cycles of MMA at N = 128). Here a tile
// of 8 x 16 output pixels loads its input window once per 64 channels, converts
// it once into shared memory (rows of 64 fp16 channels, 128-byte swizzle) and
// every tap's MMAs read it in place: pixel (py, px) of tap (ky, kx) is window row
// (stride py + ky) pitch + px + kx, so the A descriptor of a tap is the window's
// start address plus (ky pitch + kx) rows with a group stride of stride * pitch
// rows. For stride 2 the window is loaded by column parity (two units per 64
// channels), which makes the eight pixels of a group neighbours again.
//
// Exactness as in conv_kernel: chunks of whole units whose fp32 sums stay below
// 2^24 for the layer's weight codes, chunk g in accumulator region g & 1.
//
// CTA pairs (PAIR; clusters of two, cta_group::2; taken for long reductions): the
// pair takes two neighbouring M tiles of one N tile, each CTA its own window and
// accumulator rows and half of the weight columns, and the leader's MMA warp issues
// M = 256 instructions for both, so that a CTA loads and stores half the weight
// bytes.
//
// The issue is what bounds the loop over weight blocks: a wait, four MMAs, a commit
// and the counters take 240 cycles alone but 560-780 beside two epilogue warps per
// scheduler, which keep the issue slots. So a weight stage holds the taps of a
// kernel row (of one parity) where they fit, with one wait and commit for all.
//
// Persistent, one CTA per SM, 512 threads:
//   warp 0       TMA of the weight blocks (64 x n_t / 2 fp16, one per tap and unit)
//   warp 1       TMEM allocation; in the leader: MMA issue
//   warp 2       TMA of the INT8 windows
//   warps 4-11   epilogue (hatq_lean.h): with one chunk per tile the warpgroups take
//                the tiles in turn; with 128-wide groups (EPI 1128) or drains
//                (EPI 2064, 2128) both share each tile, half of every group each
//   warps 12-15  converters: INT8 window row -> fp16 window row
// Every wait is bounded, as in conv_kernel.
#include <cuda_fp16.h>

#include "hatq_internal.h"
#include "hatq_launch.h"
#include "hatq_lean.h"
#include "hatq_tc.h"

namespace hatq {
namespace {

using namespace tc;

constexpr int kThreads = 512;

// barriers from bar_off: b_full[8], b_empty[8], w8_full[2], w8_empty[2], w16_full[2],
// w16_empty[2], acc_full[4], acc_empty[4]; then the TMEM address and the abort flag.
// The leader's b_full, w16_full and acc_empty count for the pair.
constexpr int kBars = 32;

// EPI, the epilogue: 32 / 64 whole tiles per warpgroup; 1128, 2064, 2128 shared
// tiles of 128- / 64-wide groups, 2xxx with several chunks per tile: 2064 drains
// each into registers, 2128 (two chunks of 128 columns) keeps four regions;
// 3064 whole tiles with the sub-pixel rearrangement (factor 2); 4032 / 4064 whole
// tiles with the general transition (SiLU / GELU).

template <int EPI, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
    conv_win_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmY, const __grid_constant__ WinArgs a) {
    constexpr bool kSplit = EPI / 1000 == 1 || EPI / 1000 == 2, kDrain = EPI == 2064, kTwo = EPI == 2128;
    static_assert(EPI == 32 || EPI == 64 || EPI == 1128 || kDrain || kTwo || EPI == 3064 || EPI / 1000 == 4, "epilogue");
    constexpr bool kD2s = EPI / 1000 == 3, kGeneral = EPI / 1000 == 4;
    constexpr bool kQuick = !kSplit && !kGeneral;                     // fp32 estimate, exact rows where it is not certain
    constexpr int G = EPI % 1000;
    constexpr int kRegions = kTwo ? 4 : 2, kRegLog = kTwo ? 2 : 1;   // accumulator regions of n_t columns
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *bar_area = smem + a.bar_off;
    const uint32_t bar0 = smem_addr(bar_area);
    auto b_full = [&](int s) { return bar0 + 8u * s; };
    auto b_empty = [&](int s) { return bar0 + 8u * (8 + s); };
    auto w8_full = [&](int s) { return bar0 + 8u * (16 + s); };
    auto w8_empty = [&](int s) { return bar0 + 8u * (18 + s); };
    auto w16_full = [&](int s) { return bar0 + 8u * (20 + s); };
    auto w16_empty = [&](int s) { return bar0 + 8u * (22 + s); };
    auto acc_full = [&](int s) { return bar0 + 8u * (24 + s); };
    auto acc_empty = [&](int s) { return bar0 + 8u * (28 + s); };
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(bar_area + 8 * kBars);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bar_area + 8 * kBars + 4);

    // a failure already recorded ends every pair that has not started (both CTAs alike: the leader's
    // reading decides)
    __shared__ int s_skip;
    const uint32_t rank = PAIR ? blockIdx.x & 1u : 0u;   // in the pair, 0 the leader
    pdl_enter();
    if (threadIdx.x == 0) s_skip = *reinterpret_cast<volatile int *>(a.err);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = a.stages;
    if (threadIdx.x == 0) {
        for (int s = 0; s < 8; ++s) {
            mbar_init(b_full(s), 1);
            mbar_init(b_empty(s), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(w8_full(s), 1);
            mbar_init(w8_empty(s), 128);
            mbar_init(w16_full(s), PAIR ? 8 : 4);    // converter warps
            mbar_init(w16_empty(s), 1);
        }
        for (int s = 0; s < kRegions; ++s) {
            mbar_init(acc_full(s), 1);
            // epilogue warps that read the region (a tile of 32 columns is the first warpgroup's alone)
            mbar_init(acc_empty(s), (kSplit && a.n_t > G / 2 ? 8 : 4) * (PAIR ? 2 : 1));
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc512<PAIR>(smem_addr(tmem_holder));
    }
    // bias products M b (64 bits) and multipliers of all output channels, or for the fp32
    // estimate multipliers and bias products times 2^-n
    long long *mbs = reinterpret_cast<long long *>(bar_area + a.const_off);
    int *mults = reinterpret_cast<int *>(mbs + a.co);
    float *quick = reinterpret_cast<float *>(bar_area + a.const_off);
    if constexpr (kQuick) {
        stage_quick(quick, a.mult, a.b_int, a.co, a.shift);
    } else {
        for (int c = threadIdx.x; c < a.co; c += kThreads) {
            const int m = a.mult[c];
            mbs[c] = (long long)m * a.b_int[c];
            mults[c] = m;
        }
    }
    int8_t *lut_s = reinterpret_cast<int8_t *>(mults + a.co);
    if constexpr (kGeneral)
        for (int i = threadIdx.x; i < 256; i += kThreads) lut_s[i] = a.lut[i];
    tc_fence_before();
    group_sync<PAIR>();                              // both CTAs' barriers are initialized
    tc_fence_after();
    const uint32_t tmem = *tmem_holder;
    int skip = s_skip;
    if constexpr (PAIR)
        asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(skip) : "r"(leader_addr(smem_addr(&s_skip))) : "memory");
    if (skip != 0) {
        group_sync<PAIR>();                          // the leader's word has been read
        if (warp == 1) tmem_dealloc512<PAIR>(tmem);
        return;
    }

    // pair tile t: M tiles 2 (t / n_tiles_n) + rank (the last may lie past the last image: its
    // window reads zeros and nothing of it is stored), N tile t % n_tiles_n
    const int pair = (int)blockIdx.x >> (PAIR ? 1 : 0), pairs = (int)gridDim.x >> (PAIR ? 1 : 0);
    const int my_tiles = a.num_tiles > pair ? (a.num_tiles - 1 - pair) / pairs + 1 : 0;
    const int tiles_per_img = a.tiles_w * a.tiles_h;
    auto tile_coords = [&](int j, int &img, int &ho0, int &wo0, int &n0) {
        const int t = pair + j * pairs;
        const int pt = t / a.n_tiles_n, mt = PAIR ? 2 * pt + (int)rank : pt;
        n0 = (t - pt * a.n_tiles_n) * a.n_t;
        img = mt / tiles_per_img;
        const int rem = mt - img * tiles_per_img;
        const int ty = rem / a.tiles_w;
        ho0 = ty * 16;
        wo0 = (rem - ty * a.tiles_w) * 8;
    };

    // register split (launch 512 x 128): 56 / 200 / 200 / 56
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;" ::: "memory");
        // The issuing warps stay converged, their loops have uniform trip counts (a
        // wait that fails does not return) and their copies, MMAs and commits are
        // predicated on one lane: then counters, addresses and descriptors live in
        // uniform registers. Measured on h1 (3x3 320 -> 640): as branches in one
        // lane 1123 us, predicated 918 us.
        const uint32_t lead = elect_one() ? 1u : 0u;
        if (warp == 0) {
            // ------------------------------------------------------ weight producer
            // each CTA loads its half of the columns; both halves count on the leader's barrier
            const uint32_t st0 = smem_addr(smem), bytes = (uint32_t)a.b_bytes;
            const uint32_t bars = b_empty(0), bars_end = b_empty(S);
            const uint32_t to_full = (PAIR ? leader_addr(b_full(0)) : b_full(0)) - b_empty(0);   // b_empty here -> the leader's b_full
            const uint32_t expect = rank == 0 ? lead : 0u;
            const int half = (int)rank * (a.n_t / 2);
            const uint32_t st_step = bytes * (uint32_t)a.seg;
            uint32_t ph = 1, st = st0, bar = bars;
            // one stage: m blocks whose weight columns start at k, k + dk, ...
            auto load = [&](int k, int dk, int m, int n0) {
                mbar_wait_issue<PAIR>(bar, ph, abort_flag, a.err, tmem, false);
                mbar_expect_tx_if(expect, bar - 64u, (PAIR ? 2u : 1u) * bytes * (uint32_t)m);
                uint32_t dst = st;
#pragma unroll 1
                for (int i = 0; i < m; ++i, k += dk, dst += bytes)
                    if constexpr (PAIR) tma_load_2d_pair_if(lead, dst, &tmB, bar + to_full, k, n0 + half);
                    else tma_load_2d_if(lead, dst, &tmB, bar - 64u, k, n0);
                st += st_step;
                bar += 8u;
                if (bar == bars_end) { bar = bars; ph ^= 1u; st = st0; }
            };
            const int dk = a.par * a.k_tap;                  // weight columns between a row's taps
            for (int j = 0; j < my_tiles; ++j) {
                int img, ho0, wo0, n0;
                tile_coords(j, img, ho0, wo0, n0);
                if (a.pairs) {
                    for (int i = 0; i < a.kblocks; i += a.seg) load(i * 64, 64, min(a.seg, a.kblocks - i), n0);
                    continue;
                }
                for (int cb = 0; cb < a.cin_kb; ++cb)
                    for (int p = 0; p < a.par; ++p)
                    {
                        const int taps = a.par == 2 ? (a.kw - p + 1) >> 1 : a.kw;        // of a kernel row
                        int k = p * a.k_tap + cb * 64;
                        for (int ky = 0; ky < a.kh; ++ky, k += a.kw * a.k_tap)
                            for (int t = 0; t < taps; t += a.seg)
                                load(k + t * dk, dk, min(a.seg, taps - t), n0);
                    }
            }
        } else if (warp == 2) {
            // ------------------------------------------------------ window producer
            int s = 0;
            uint32_t ph = 1;
            for (int j = 0; j < my_tiles; ++j) {
                int img, ho0, wo0, n0;
                tile_coords(j, img, ho0, wo0, n0);
                const int x0 = wo0 * a.stride - a.pad_x, y0 = ho0 * a.stride - a.pad_y;
                for (int cb = 0; cb < a.cin_kb; ++cb)
                    for (int p = 0; p < a.par; ++p) {
                        mbar_wait_issue<PAIR>(w8_empty(s), ph, abort_flag, a.err, tmem, false);
                        mbar_expect_tx_if(lead, w8_full(s), (uint32_t)(a.rows * 64));
                        tma_load_4d_if(lead, smem_addr(smem) + (uint32_t)(a.w8_off + s * a.w8_bytes), &tmA, w8_full(s), cb * 64,
                                       x0 + p, y0, img);
                        if (++s == a.n8) { s = 0; ph ^= 1u; }
                    }
            }
        } else if (warp == 1 && rank == 0) {
            // ------------------------------------------------------ MMA issuer
            const uint32_t idesc = idesc_f16(a.n_t, PAIR ? 256 : 128);
            // descriptor halves: start address (and the unused leading offset) in the low word; group
            // stride, version and 128-byte swizzle in the high word
            const uint32_t bhi = (1024u >> 4) | (1u << 14) | (2u << 29);
            const uint32_t ahi = (uint32_t)((a.stride * a.pitch * 128) >> 4) | (1u << 14) | (2u << 29);
            const uint32_t blo0 = ((smem_addr(smem) >> 4) & 0x3FFFu) | (1u << 16);
            const uint32_t alo0 = ((smem_addr(smem + a.w16_off) >> 4) & 0x3FFFu) | (1u << 16);
            const uint32_t b_step = (uint32_t)a.b_bytes >> 4, w_step = (uint32_t)a.w16_bytes >> 4;
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
            int ws = 0, g = 0;
            uint32_t ph = 0, wph = 0, acc = 0, d = tm;
            uint32_t bl = blo0;                              // the weight stage's descriptor
            const uint32_t st_step = b_step * (uint32_t)a.seg, row_step = (uint32_t)(a.pitch * 8);
            uint32_t bar = b_full(0);                        // b_full of the stage; its b_empty is 64 bytes on
            const uint32_t bar_end = b_full(S);
            // one weight block: K steps 0-1 read the window at o0, 2-3 at o1 (nk of them)
            auto block = [&](uint32_t o0, uint32_t o1, uint32_t b, int nk) {
                umma_f16_ss_if<PAIR>(lead, d, o0, ahi, b, bhi, idesc, acc);
                if (nk > 1) umma_f16_ss_if<PAIR>(lead, d, o0 + 2, ahi, b + 2, bhi, idesc, 1u);
                if (nk > 2) umma_f16_ss_if<PAIR>(lead, d, o1, ahi, b + 4, bhi, idesc, 1u);
                if (nk > 3) umma_f16_ss_if<PAIR>(lead, d, o1 + 2, ahi, b + 6, bhi, idesc, 1u);
                acc = 1u;
            };
            auto stage_done = [&]() {
                umma_commit_if<PAIR>(lead, bar + 64u);
                bl += st_step;
                bar += 8u;
                if (bar == bar_end) { bar = b_full(0); ph ^= 1u; bl = blo0; }
            };
            // one stage of a kernel row: m taps from window offset o on
            auto row = [&](uint32_t o, int m, int nk) {
                mbar_wait_issue<PAIR>(bar, ph, abort_flag, a.err, tm, true);
                uint32_t b = bl;
#pragma unroll 1
                for (int i = 0; i < m; ++i, o += 8, b += b_step) block(o, o + 4, b, nk);
                stage_done();
            };
            for (int j = 0; j < my_tiles; ++j) {
                int left = a.cin_kb * a.par;                 // units left in the tile
                int cu = 0;                                  // units of the current chunk
                for (int cb = 0; cb < a.cin_kb; ++cb)
                    for (int p = 0; p < a.par; ++p) {
                        if (cu == 0) {
                            const int reg = g & (kRegions - 1);
                            d = tm + (uint32_t)(reg * a.n_t);
                            acc = 0u;
                            if (g >= kRegions)
                                mbar_wait_issue<PAIR>(acc_empty(reg), ((g >> kRegLog) - 1) & 1, abort_flag, a.err, tm, true);
                        }
                        mbar_wait_issue<PAIR>(w16_full(ws), wph, abort_flag, a.err, tm, true);
                        tc_fence_after();
                        const uint32_t w0 = alo0 + (uint32_t)ws * w_step;
                        if (a.pairs) {
                            // two 32-channel taps per weight block (64 bytes of each window row are zero)
                            int ky = 0, kx = 0;
                            for (int i0 = 0; i0 < a.kblocks; i0 += a.seg) {
                                mbar_wait_issue<PAIR>(bar, ph, abort_flag, a.err, tm, true);
                                uint32_t b = bl;
                                const int m = min(a.seg, a.kblocks - i0);
#pragma unroll 1
                                for (int i = 0; i < m; ++i, b += b_step) {
                                    const uint32_t o0 = w0 + (uint32_t)((ky * a.pitch + kx) * 8);
                                    if (++kx == a.kw) { kx = 0; ++ky; }
                                    const int nk = ky < a.kh ? 4 : 2;
                                    const uint32_t o1 = w0 + (uint32_t)((ky * a.pitch + kx) * 8);
                                    if (++kx == a.kw) { kx = 0; ++ky; }
                                    block(o0, o1, b, nk);
                                }
                                stage_done();
                            }
                        } else {
                            const int taps = a.par == 2 ? (a.kw - p + 1) >> 1 : a.kw;    // of a kernel row
                            const int nk = cb == a.cin_kb - 1 ? a.nk_last : 4;
                            uint32_t orow = w0;
                            for (int ky = 0; ky < a.kh; ++ky, orow += row_step)
                                for (int t = 0; t < taps; t += a.seg)
                                    row(orow + (uint32_t)(8 * t), min(a.seg, taps - t), nk);
                        }
                        umma_commit_if<PAIR>(lead, w16_empty(ws));
                        if (++ws == 2) { ws = 0; wph ^= 1u; }
                        --left;
                        if (++cu == a.chunk_units || left == 0) {
                            umma_commit_if<PAIR>(lead, acc_full(g & (kRegions - 1)));
                            ++g;
                            cu = 0;
                        }
                    }
            }
            // (the epilogues end after the last chunk's commit, which covers every MMA)
        }
    } else if (warp >= 12) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;" ::: "memory");
        // ---------------------------------------------------------- converters
        const int row0 = ((int)threadIdx.x - 384) >> 2, q4 = (int)threadIdx.x & 3;
        bool ok = true;
        int s8 = 0, s16 = 0;
        uint32_t p8 = 0, p16 = 0;
        const int total = my_tiles * a.cin_kb * a.par;
        for (int u = 0; u < total; ++u) {
            ok = __all_sync(0xffffffffu, mbar_wait(w8_full(s8), p8, abort_flag, a.err));
            if (ok) ok = __all_sync(0xffffffffu, mbar_wait(w16_empty(s16), p16 ^ 1u, abort_flag, a.err));
            if (!ok) break;
            const uint8_t *src = smem + a.w8_off + s8 * a.w8_bytes;
            uint8_t *dst = smem + a.w16_off + s16 * a.w16_bytes;
            // 16 codes (64-byte swizzle) -> 16 fp16 values (128-byte swizzle) per step; a thread keeps
            // its quarter of the row and moves on by 32 rows, so its swizzle terms stay the same
            const uint8_t *sp = src + row0 * 64 + ((q4 ^ ((row0 >> 1) & 3)) << 4);
            uint8_t *dp = dst + row0 * 128;
            const int d0 = ((2 * q4) ^ (row0 & 7)) << 4, d1 = ((2 * q4 + 1) ^ (row0 & 7)) << 4;
            auto convert = [&](const uint4 &v, uint8_t *out) {
                uint4 lo, hi;
                i8x4_to_f16x4(v.x, lo.x, lo.y);
                i8x4_to_f16x4(v.y, lo.z, lo.w);
                i8x4_to_f16x4(v.z, hi.x, hi.y);
                i8x4_to_f16x4(v.w, hi.z, hi.w);
                *reinterpret_cast<uint4 *>(out + d0) = lo;
                *reinterpret_cast<uint4 *>(out + d1) = hi;
            };
            int r = row0;
#pragma unroll 1
            for (; r + 64 < a.rows; r += 96, sp += 96 * 64, dp += 96 * 128) {
                const uint4 v0 = *reinterpret_cast<const uint4 *>(sp), v1 = *reinterpret_cast<const uint4 *>(sp + 32 * 64);
                const uint4 v2 = *reinterpret_cast<const uint4 *>(sp + 64 * 64);
                convert(v0, dp);
                convert(v1, dp + 32 * 128);
                convert(v2, dp + 64 * 128);
            }
#pragma unroll 1
            for (; r < a.rows; r += 32, sp += 32 * 64, dp += 32 * 128) convert(*reinterpret_cast<const uint4 *>(sp), dp);
            fence_async_shared();                    // the MMAs read the window through the async proxy
            __syncwarp();
            if (lane == 0) {
                if constexpr (PAIR) mbar_arrive_cluster(leader_addr(w16_full(s16)));
                else mbar_arrive(w16_full(s16));
            }
            mbar_arrive(w8_empty(s8));
            if (++s8 == a.n8) { s8 = 0; p8 ^= 1u; }
            if (++s16 == 2) { s16 = 0; p16 ^= 1u; }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 200;" ::: "memory");
        // ---------------------------------------------------------- epilogue (warps 4-11)
        const int wg = (warp - 4) >> 2;            // 0 or 1
        const int quad = warp & 3;                 // TMEM lane quadrant this warp may access
        const uint32_t t_lane = tmem + ((uint32_t)(quad * 32) << 16);
        uint8_t *staging = smem + a.stg_off;
        uint8_t *wstage = staging + (warp - 4) * kWarpStage;
        bool ok = true;
        int buf = 0;
        [[maybe_unused]] const Quick opt = quick_setup<G>(a.hb_out, a.hb_next, a.act, a.shift);
        // this warp's tensor-memory reads of a region are done (fenced by every lane)
        auto release = [&](int r) {
            __syncwarp();
            if (lane == 0) {
                if constexpr (PAIR) mbar_arrive_cluster(leader_addr(acc_empty(r)));
                else mbar_arrive(acc_empty(r));
            }
        };
        for (int j = 0; j < my_tiles; ++j) {
            if (!kSplit && (j & 1) != wg) continue;
            int img, ho0, wo0, n0;
            tile_coords(j, img, ho0, wo0, n0);
            const int oy = ho0 + 4 * quad, ox = wo0;       // this warp's 32 rows: 4 x 8 pixels
            const bool inside = oy < a.ho && ox < a.wo && img < a.n;
            if constexpr (!kSplit) {
                const int reg = j & 1;
                const uint32_t t_acc = t_lane + (uint32_t)(reg * a.n_t);
                ok = __all_sync(0xffffffffu, mbar_wait(acc_full(reg), (j >> 1) & 1, abort_flag, a.err));
                tc_fence_after();
                if (!ok) break;
#pragma unroll 1
                for (int col = 0; col < a.n_t; col += G) {
                    uint32_t r[G], w[G / 4];
#pragma unroll
                    for (int q = 0; q < G / 32; ++q)
                        tmem_ld32(t_acc + col + 32 * q, reinterpret_cast<uint32_t(&)[32]>(r[32 * q]));
                    tmem_wait_ld();
                    if (col + G >= a.n_t) {                                // TMEM reads of this region are complete
                        tc_fence_before();
                        release(reg);
                    }
                    if constexpr (kGeneral) {
                        // z = clamp(round(H~_out (M_out (.) a) / 2^n_out)), u = phi_int(z), then the next
                        // layer's transform on u itself (|H~ u| <= 127 * 64) and its requantization
                        long long t[G];
                        lean_scale<G>(r, mbs + n0 + col, mults + n0 + col, t);
                        if (a.hb_out) fwht_stages<G>(t, a.hb_out);
                        int u[G];
#pragma unroll
                        for (int i = 0; i < G; ++i) u[i] = (int)lut_s[requant8_any(t[i], a.shift) + 127];
                        if (a.hb_next) fwht_stages<G>(u, a.hb_next);
#pragma unroll
                        for (int i = 0; i < G / 4; ++i) {
                            int q[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) q[k] = requant8_any(a.mult_in * (long long)u[4 * i + k], a.shift_in);
                            w[i] = pack4(q[0], q[1], q[2], q[3]);
                        }
                    } else {
                        const float *ms = quick + n0 + col;
                        const bool sure = quick_codes<G>(r, ms, ms + a.co, opt, lane, w);
                        const uint32_t rows = __ballot_sync(0xffffffffu, !sure);
                        if (rows)
                            exact_rows<G>(rows, r, reinterpret_cast<const int *>(ms) + 2 * a.co,
                                          reinterpret_cast<const int *>(ms) + 3 * a.co, opt,
                                          staging + 8 * kWarpStage + (warp - 4) * kWarpScratch, lane, w);
                    }
                    if constexpr (kD2s) {
                        // channel 4 cd + 2 i + j of this lane's pixel -> channel cd of pixel (2 oy + i, 2 ox + j):
                        // word k holds the four codes of one cd, so 4 x 4 byte transposes give 16 channels
                        // of each of the four pixels
                        uint32_t o[4][4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint32_t t0 = __byte_perm(w[4 * q], w[4 * q + 1], 0x5140);
                            const uint32_t t1 = __byte_perm(w[4 * q + 2], w[4 * q + 3], 0x5140);
                            const uint32_t t2 = __byte_perm(w[4 * q], w[4 * q + 1], 0x7362);
                            const uint32_t t3 = __byte_perm(w[4 * q + 2], w[4 * q + 3], 0x7362);
                            o[0][q] = __byte_perm(t0, t1, 0x5410);
                            o[1][q] = __byte_perm(t0, t1, 0x7632);
                            o[2][q] = __byte_perm(t2, t3, 0x5410);
                            o[3][q] = __byte_perm(t2, t3, 0x7632);
                        }
                        const int py = oy + (lane >> 3), px = ox + (lane & 7);
                        if (py < a.ho && px < a.wo && img < a.n) {
                            uint8_t *y = static_cast<uint8_t *>(a.y) + (n0 + col) / 4 +
                                         (((long long)img * a.ho + py) * 4 * a.wo + 2 * px) * (a.co / 4);
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                *reinterpret_cast<uint4 *>(y + (long long)((k >> 1) * 2 * a.wo + (k & 1)) * (a.co / 4)) =
                                    make_uint4(o[k][0], o[k][1], o[k][2], o[k][3]);
                        }
                    } else {
                        lean_store<G>(wstage + buf * (kWarpStage / 2), w, &tmY, lane, inside, n0 + col, ox, oy, img);
                        buf ^= 1;
                    }
                }
            } else {
                constexpr int H = G / 2;                   // columns of a group this warp finishes
                constexpr int NP = G == 64 ? 3 : 1;        // groups of a tile (n_t <= 192 / n_t = 128)
                const uint8_t *theirs = staging + (wg ? warp - 8 : warp) * kWarpStage;
                uint32_t part[kDrain ? NP : 1][kDrain ? H : 1];   // exact int32 sums of the drained chunks
                // groups of this warp: columns (2 gr + wg) H .. + H - 1 (tiles of 32-wide groups may hold an odd number)
                const int ng = (a.n_t / H - wg + 1) / 2;
                if (ng == 0) continue;                     // n_t = 32: the other warpgroup has the tile to itself
                for (int ch = 0; kDrain && ch + 1 < a.nch; ++ch) {
                    const int gc = j * a.nch + ch, reg = gc & 1;
                    if (ok) ok = __all_sync(0xffffffffu, mbar_wait(acc_full(reg), (gc >> 1) & 1, abort_flag, a.err));
                    tc_fence_after();
                    if (ok) {
#pragma unroll
                        for (int gr = 0; gr < NP; ++gr) {
                            if (gr >= ng) break;
#pragma unroll
                            for (int q = 0; q < H / 32; ++q) {
                                uint32_t r[32];
                                tmem_ld32(t_lane + (uint32_t)(reg * a.n_t + gr * G + wg * H + 32 * q), r);
                                tmem_wait_ld();
#pragma unroll
                                for (int i = 0; i < 32; ++i) {
                                    const uint32_t v = (uint32_t)__float2int_rn(__uint_as_float(r[i]));
                                    if constexpr (kDrain) part[gr][32 * q + i] = ch ? part[gr][32 * q + i] + v : v;
                                }
                            }
                        }
                    }
                    tc_fence_before();
                    release(reg);
                }
                // the last chunk's region; with 2128 both chunks of the tile still sit in regions of their own
                const int gc = j * a.nch + a.nch - 1, reg = gc & (kRegions - 1), reg0 = (gc - 1) & (kRegions - 1);
                if constexpr (kTwo)
                    if (ok) ok = __all_sync(0xffffffffu, mbar_wait(acc_full(reg0), ((gc - 1) >> kRegLog) & 1, abort_flag, a.err));
                if (ok) ok = __all_sync(0xffffffffu, mbar_wait(acc_full(reg), (gc >> kRegLog) & 1, abort_flag, a.err));
                tc_fence_after();
                // one copy of this code for all groups: unrolled it would not fit the instruction cache
#pragma unroll 1
                for (int gr = 0; gr < ng; ++gr) {
                    const int col = gr * G + wg * H;
                    long long t[H];
#pragma unroll
                    for (int q = 0; q < H / 32; ++q) {
                        uint32_t r[32], r0[kTwo ? 32 : 1];
                        tmem_ld32(t_lane + (uint32_t)(reg * a.n_t + col + 32 * q), r);
                        if constexpr (kTwo) tmem_ld32(t_lane + (uint32_t)(reg0 * a.n_t + col + 32 * q), r0);
                        tmem_wait_ld();
                        if (q == H / 32 - 1 && gr == ng - 1) {
                            tc_fence_before();
                            release(reg);
                            if constexpr (kTwo) release(reg0);
                        }
                        const long long *mb = mbs + n0 + col + 32 * q;
                        const int *mu = mults + n0 + col + 32 * q;
#pragma unroll
                        for (int i = 0; i < 32; i += 4) {
                            const int4 m = *reinterpret_cast<const int4 *>(mu + i);
                            const longlong2 b0 = *reinterpret_cast<const longlong2 *>(mb + i);
                            const longlong2 b1 = *reinterpret_cast<const longlong2 *>(mb + i + 2);
                            int v[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                v[k] = __float2int_rn(__uint_as_float(r[i + k]));
                                if constexpr (kDrain)     // (selected, as registers have no index)
                                    v[k] += (int)(gr == 0 ? part[0][i + k] : (gr == 1 ? part[1][i + k] : part[2][i + k]));
                                if constexpr (kTwo) v[k] += __float2int_rn(__uint_as_float(r0[i + k]));
                            }
                            t[32 * q + i] = (long long)m.x * v[0] + b0.x;
                            t[32 * q + i + 1] = (long long)m.y * v[1] + b0.y;
                            t[32 * q + i + 2] = (long long)m.z * v[2] + b1.x;
                            t[32 * q + i + 3] = (long long)m.w * v[3] + b1.y;
                        }
                    }
                    split_finish<G>(t, a.shift, a.hb_out, a.hb_next, a.act, wstage, theirs, wg, quad, lane, &tmY,
                                    inside && ok, n0 + col, ox, oy, img);
                }
            }
        }
        if (lane == 0) bulk_wait_all();
    }

    tc_fence_before();
    group_sync<PAIR>();                              // nothing of the other CTA reaches this one any more
    tc_fence_after();
    if (warp == 1) tmem_dealloc512<PAIR>(tmem);
}

}  // namespace

cudaError_t launch_conv_win(const CUtensorMap &tmA, const CUtensorMap &tmB, const CUtensorMap &tmY, const WinArgs &a, int epi,
                            int smem_bytes, cudaStream_t s) {
    using Fn = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const WinArgs);
#define HATQ_WIN(e) {e, {conv_win_kernel<e, false>, conv_win_kernel<e, true>}}
    static const struct { int epi; Fn fn[2]; } kerns[] = {HATQ_WIN(32),   HATQ_WIN(64),   HATQ_WIN(1128), HATQ_WIN(2064),
                                                          HATQ_WIN(2128), HATQ_WIN(3064), HATQ_WIN(4032), HATQ_WIN(4064)};
#undef HATQ_WIN
    constexpr int kKerns = sizeof(kerns) / sizeof(kerns[0]);
    int v = 0;
    while (v < kKerns && kerns[v].epi != epi) ++v;
    if (v == kKerns) return cudaErrorInvalidValue;
    const int pr = a.pair ? 1 : 0;
    const Fn kern = kerns[v].fn[pr];
    static SmemOptIn opt_in[kKerns][2];
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = current_device(&dev)) != cudaSuccess || (e = opt_in[v][pr].set(dev, reinterpret_cast<const void *>(kern))) != cudaSuccess ||
        (e = device_sms(dev, &sms)) != cudaSuccess)
        return e;
    const int groups = pr ? (sms / 2 < 1 ? 1 : sms / 2) : sms;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((pr ? 2 : 1) * (a.num_tiles < groups ? a.num_tiles : groups));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1 + pr;
    return cudaLaunchKernelEx(&cfg, kern, tmA, tmB, tmY, a);
}

}  // namespace hatq
