// Digit-plane products of less than two waves of tiles: the tiles' sums go to
// memory and a separate finish pass applies the step.
//
// In the persistent product kernel (digits_kernel.cuh) the epilogue of a 128 x
// 128 tile is done by the tile's own eight warps: 28 us or more in which, when
// every CTA has one tile, the tensor pipe is idle, and with few tiles most SMs
// too (n = 200: three tiles, 67 us per product for 8 us of MMAs).  Here the CTA of
// a tile, or of a part of a tile of the split last wave, only empties its
// accumulators: levels 0 to 2 as exact integers, added to one 64-bit word per
// element (atomically, where a tile has parts), the shared accumulator of levels
// >= 3 as floats, one array per part.  A second kernel spreads the polynomial, the
// re-split and the stores over all SMs in 32 x 32 blocks.  The two overlap their
// prologues (programmatic stream serialization).
//
// The work items (whole tiles, and the parts of digit_split_plan), the sums and
// the order in which a finish adds the parts are those of the persistent
// kernel, so the densities are the same bit for bit.
//
// A leading level that is not finite or out of any iterate's range (2^20: a
// product's entry of 16 where iterates stay below 1; the sum of a tile's four
// parts still fits) poisons the run: the finish pass writes NaN from then on, and
// the caller runs it again on the persistent kernel, which carries such values.
//
// Measured per product of a run, host calls included (persistent kernel -> here):
// n = 200 67 -> 17 us, n = 1101 92 -> 38 us, n = 2000 at 5 digits 130 -> 110 us, n =
// 2500 258 -> 195 us, n = 2900 288 -> 275 us (nearly two full waves).  From two
// waves on the persistent kernel's queue launches overlap one tile's epilogue
// with the next tile's MMAs.
#include <algorithm>
#include <mutex>

#include "digits_fixed.h"
#include "digits_kernel.cuh"
#include "tile_sums.cuh"

namespace purify {

using namespace dk;

int fill_digit_params(const DigitStep& st, DigitGemmParams* p, CUtensorMap* ma, CUtensorMap* mb);  // digits_tc.cu

namespace {

// 16 epilogue warps, each 32 rows x 32 columns of a tile: with 8 an emptying of the
// accumulators waits on its own arithmetic (two warps per scheduler)
constexpr int kEpi = 16;
constexpr int kThreads = 64 + 32 * kEpi;
constexpr int kMaxRegs = 96;  // 18 warps: five on a sub-partition of 16384 registers

struct FixedLaunch {
    CUtensorMap map_a, map_b;
    DigitGemmParams prm;
    FixedSums sums;
    int* err;
    long long wait_cycles;
    int items, split_begin, ways;
    int halves;  // 2: an item's levels 0..2 (half 0) and levels >= 3 (half 1) on two CTAs
};

// Unit u of the grid: an item, or one of its halves.
__device__ __forceinline__ int fixed_unit(const FixedLaunch& L, int u, int& half) {
    half = u >= L.items;
    return half ? u - L.items : u;
}

// Work item t: a tile, or a part of a tile of the last wave; and the k-chunks
// it sums.  Item t's share of levels >= 3 is sums.shared[t].
__device__ __forceinline__ void fixed_item(const FixedLaunch& L, int t, int& ti, int& tj, int& k0, int& count) {
    const int nk = L.prm.tiles_per_row * 4;
    int tile = t;
    k0 = 0;
    count = nk;
    if (t >= L.split_begin) {
        const int u = t - L.split_begin, slot = u / L.ways, part = u - slot * L.ways;
        tile = L.split_begin + slot;
        k0 = part * nk / L.ways;
        count = (part + 1) * nk / L.ways - k0;
    }
    decode_banded(tile, L.prm.tiles_per_row, ti, tj);
}

// The number that decode_banded takes to (ti, tj).
__device__ __forceinline__ int encode_banded(int ti, int tj, int T) {
    const int b0 = tj / BAND * BAND, b1 = min(T, b0 + BAND);
    const int below = min(ti, b0), r = max(ti - b0, 0);  // rows above b0, and from b0 on
    return b0 * (b0 + 1) / 2 + below * (b1 - b0) + r * (b1 - b0) - r * (r - 1) / 2 + tj - max(b0, ti);
}

// Levels 0 and 1 (units of 2^-7, high word) and 2 (units of 2^-14, low word) of
// one element as a 64-bit integer: sums of such words hold the sums of both.
template <int NA>
__device__ __forceinline__ unsigned long long pack_levels(float a0, float a1, float a2) {
    int h = (int)(__float_as_uint(a0 + kMagic) - kMagicBits) << 7, l = 0;
    if (NA > 1) h += (int)(__float_as_uint(fmaf(a1, 128.f, kMagic)) - kMagicBits);
    if (NA > 2) {  // below 2^24: in two pieces
        const float v = a2 * 16384.f, t = fmaf(v, 1.f / 4096.f, kMagic), r = fmaf(t - kMagic, -4096.f, v) + kMagic;
        l = ((int)(__float_as_uint(t) - kMagicBits) << 12) + (int)(__float_as_uint(r) - kMagicBits);
    }
    return (unsigned long long)(unsigned int)(h + (l >> 31)) << 32 | (unsigned int)l;
}

// The MMAs of one 32-wide k-chunk for levels 0..2 (HALF 0) or for the shared
// accumulator of levels >= 3 (HALF 1), each accumulator's in issue_chunk's order.
template <int S, int HALF>
__device__ __forceinline__ void issue_half(uint32_t tmem, uint64_t da, uint64_t db, uint32_t later) {
#pragma unroll
    for (int p = 0; p < S; ++p)
#pragma unroll
        for (int q = 0; q < S - p; ++q) {
            if ((p + q >= NUM_ACC - 1) != (HALF == 1)) continue;
            const int a = HALF ? NUM_ACC - 1 : p + q;
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
                mma_bf16(tmem + (uint32_t)(a * TILE), da + (uint64_t)plane_desc_off(p, kk),
                         db + (uint64_t)plane_desc_off(q, kk), IDESC, (kk > 0 || p > 0 || q > NUM_ACC - 1) ? 1u : later);
        }
}

template <int S>
constexpr int fixed_stages() {
    constexpr int n = (200 * 1024) / (2 * plane_pairs(S) * PAIR_BYTES);
    return n < 4 ? n : 4;
}
template <int S>
constexpr int fixed_smem() {
    return 1024 + fixed_stages<S>() * 2 * plane_pairs(S) * PAIR_BYTES + 256;
}

// The issue order of issue_chunk (digits_kernel.cuh): one stage is a 32-wide
// k-chunk of both operands' S planes.
template <int S>
__global__ void __maxnreg__(kMaxRegs) digit_fixed_kernel(const __grid_constant__ FixedLaunch L) {
    constexpr int NP = plane_pairs(S), kStages = fixed_stages<S>(), kStageBytes = 2 * NP * PAIR_BYTES;
    constexpr int NA = S < NUM_ACC ? S : NUM_ACC;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full_bar = (uint64_t*)(base + kStages * kStageBytes);
    uint64_t* empty_bar = full_bar + kStages;
    uint64_t* tmem_full = empty_bar + kStages;
    uint64_t* tmem_empty = tmem_full + 1;
    uint64_t* drain = tmem_full + 2;
    uint32_t* tmem_slot = (uint32_t*)(drain + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long wait = L.wait_cycles > 0 ? L.wait_cycles : WAIT_CYCLES;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * kStages; ++i) mbar_init(smem_u32(&full_bar[i]), 1);
        mbar_init(smem_u32(tmem_full), 1);
        mbar_init(smem_u32(tmem_empty), kEpi);
        mbar_init(smem_u32(drain), 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), NUM_ACC * TILE);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    int ti, tj, k0, count, half;
    grid_dependency_wait();
    // a step controlled on the device (uniform over the grid: written by an earlier kernel)
    const DevStep* ctl = L.prm.ctl;
    const bool skip = ctl && (ctl->done || ctl->s_in != S);

    if (skip) {
    } else if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            for (int u = blockIdx.x; ok && u < L.items * L.halves; u += gridDim.x) {
                fixed_item(L, fixed_unit(L, u, half), ti, tj, k0, count);
                for (int c = 0; c < count; ++c, ++it) {
                    const int st = it % kStages;
                    if ((it >= kStages &&
                         !mbar_wait_for(smem_u32(&empty_bar[st]), (uint32_t)(((it / kStages) & 1) ^ 1), wait)) ||
                        *abort_flag) {
                        ok = false;
                        break;
                    }
                    const uint32_t fb = smem_u32(&full_bar[st]);
                    const uint32_t sa = smem_u32(base + (size_t)st * kStageBytes);
                    mbar_arrive_expect_tx(fb, (uint32_t)kStageBytes);
                    tma_load_3d(sa, &L.map_a, fb, (k0 + c) * 64, ti * TILE, 0);
                    tma_load_3d(sa + NP * PAIR_BYTES, &L.map_b, fb, (k0 + c) * 64, tj * TILE, 0);
                }
            }
            if (!ok) {
                atomicOr(L.err, ERR_PRODUCER_WAIT);
                *abort_flag = 1;
            }
            // wait (bounded) for the copies still in flight
            for (int k = (it > kStages ? it - kStages : 0); k < it; ++k)
                mbar_wait_for(smem_u32(&full_bar[k % kStages]), (uint32_t)((k / kStages) & 1));
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint64_t desc_base = smem_desc(smem_u32(base));
            int it = 0;
            bool ok = true;
            for (int u = blockIdx.x, lt = 0; ok && u < L.items * L.halves; u += gridDim.x, ++lt) {
                fixed_item(L, fixed_unit(L, u, half), ti, tj, k0, count);
                if (lt > 0 && !mbar_wait_for(smem_u32(tmem_empty), (uint32_t)((lt - 1) & 1), wait)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                for (int c = 0; c < count; ++c, ++it) {
                    const int st = it % kStages;
                    if (!mbar_wait_for(smem_u32(&full_bar[st]), (uint32_t)((it / kStages) & 1), wait)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t da = desc_base + (uint64_t)((st * kStageBytes) >> 4);
                    const uint64_t db = da + (uint64_t)((NP * PAIR_BYTES) >> 4);
                    const uint32_t later = c > 0 ? 1u : 0u;
                    if (L.halves == 1)
                        issue_chunk<S>(tmem, da, db, later);
                    else if (half)
                        issue_half<S, 1>(tmem, da, db, later);
                    else
                        issue_half<S, 0>(tmem, da, db, later);
                    mma_commit(smem_u32(&empty_bar[st]));
                }
                if (ok) mma_commit(smem_u32(tmem_full));
            }
            if (!ok) {
                atomicOr(L.err, ERR_MMA_WAIT);
                *abort_flag = 1;
            }
            mma_commit(smem_u32(drain));
            mbar_wait_for(smem_u32(drain), 0);
        }
    } else {
        // epilogue warps: lane quarter warp % 4, the (warp - 2) / 4-th 32 columns
        const int quarter = warp & 3, col0 = ((warp - 2) >> 2) * (TILE * 4 / kEpi);
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)col0;
        bool bad = false;
        for (int u = blockIdx.x, lt = 0; u < L.items * L.halves; u += gridDim.x, ++lt) {
            const int t = fixed_unit(L, u, half);
            const bool exact = !half, rest = NA > 3 && (half || L.halves == 1);
            fixed_item(L, t, ti, tj, k0, count);
            bool ready = mbar_wait_for(smem_u32(tmem_full), (uint32_t)(lt & 1), wait);
            if (!ready) {
                atomicOr(L.err, ERR_EPI_WAIT);
                *abort_flag = 1;
            }
            ready = __all_sync(0xffffffffu, ready && !*abort_flag);  // tcgen05.ld is warp-collective
            if (!ready) break;
            tc_fence_after();
            // column-major inside a tile: a warp writes 32 consecutive values
            const int off = quarter * 32 + lane + col0 * TILE;
            const bool part = t >= L.split_begin;
            unsigned long long* sum =
                (part ? L.sums.parts + (size_t)((t - L.split_begin) / L.ways) * (TILE * TILE)
                      : L.sums.levels + (size_t)t * (TILE * TILE)) + off;
            float* shared = L.sums.shared + (size_t)t * (TILE * TILE) + off;
            uint32_t r[2][32];
            tmem_issue32(taddr, r[0]);
#pragma unroll
            for (int q = 0; q < TILE * 4 / kEpi / 8; ++q) {
                uint32_t(&v)[32] = r[q & 1];
                tmem_wait32(v);
                if (q < TILE * 4 / kEpi / 8 - 1) {
                    tmem_issue32(taddr + (uint32_t)(8 * (q + 1)), r[(q + 1) & 1]);
                } else {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(tmem_empty)) : "memory");
                }
                // blocks below the diagonal are the mirror of others
                if (ti == tj && quarter > ((col0 + 8 * q) >> 5)) continue;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (exact) {
                        const float a0 = __uint_as_float(v[c]), a1 = __uint_as_float(v[8 + c]);
                        bad |= !(fabsf(a0) < 1048576.f) || (NA > 1 && !(fabsf(a1) < 32768.f));
                        const unsigned long long x = pack_levels<NA>(a0, a1, __uint_as_float(v[16 + c]));
                        if (part)
                            atomicAdd(sum + (8 * q + c) * TILE, x);
                        else
                            sum[(8 * q + c) * TILE] = x;
                    }
                    if (rest) shared[(8 * q + c) * TILE] = __uint_as_float(v[24 + c]);
                }
            }
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) *(volatile int*)L.sums.poison = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, NUM_ACC * TILE);
    }
}

// s + x, out of line: float64 instructions whose predicate is off still take
// their turn on that pipe, and few elements need one.
__device__ __noinline__ double add_df(double s, df x) { return s + (double)x.h + (double)x.l; }

constexpr int FC = 4;  // columns of one thread

// Finish: 32 x 32 blocks I <= J of the padded matrix, lane = row, warp w =
// columns 4w .. 4w + 3 of the block.  The polynomial and the re-split are those of
// digits_kernel.cuh's phase 2.  The mirror block (and a diagonal block's both
// halves) goes through shared memory, so that planes are written in 16-byte
// pieces on both sides.  Latency-bound at small n (n = 200: 28 blocks); at n = 2048
// about 100 bytes per upper element from and to L2 / HBM.
template <int S>
__global__ void __launch_bounds__(256, 4)
digit_finish_kernel(const __grid_constant__ DigitGemmParams P, const FixedSums sums, int split_begin, int ways, int blocks) {
    constexpr int NA = S < NUM_ACC ? S : NUM_ACC;
    // digits by [plane][row][column] of the block and of its mirror, rows padded to 80 bytes
    __shared__ __align__(16) unsigned short dir[kMaxDigitPlanes][32][40], mir[kMaxDigitPlanes][32][40];
    __shared__ float rsum[2][8];
    grid_dependency_wait();
    const DevStep* ctl = P.ctl;
    if (ctl && (ctl->done || ctl->s_in != S)) return;
    const bool bad = *(volatile int*)sums.poison != 0;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int n = P.n, n_pad = P.n_pad, two_np = 2 * n_pad;
    const size_t pair_stride = (size_t)two_np * n_pad;
    df cP = P.cP, cE = P.cE, cI = P.cI;
    int s_out = P.s_out;
    __nv_bfloat16* outp = P.out;
    double* out64 = P.out64;
    if (ctl) {
        cP = dev_df(ctl->cP);
        cE = dev_df(ctl->cE);
        cI = dev_df(ctl->cI);
        s_out = ctl->s_out;
        if (s_out == 0) outp = nullptr;
        if (!ctl->write64) out64 = nullptr;
    }
    const bool use_E = P.use_E, affine = P.affine_out, want_red = P.red != nullptr;
    double s_tr = 0.0;
    float s_idem = 0.f, s_fro = 0.f;
    for (int b = blockIdx.x; b < blocks; b += gridDim.x) {
        int J = (int)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
        while ((J + 1) * (J + 2) / 2 <= b) ++J;
        while (J * (J + 1) / 2 > b) --J;
        const int I = b - J * (J + 1) / 2;
        const bool diag = I == J;
        const int i = I * 32 + lane, j0 = J * 32 + FC * w;
        const int off = ((J & 3) * 32 + FC * w) * TILE + (I & 3) * 32 + lane;
        const int tile = encode_banded(I >> 2, J >> 2, P.tiles_per_row);
        const bool split = tile >= split_begin;
        unsigned long long* t = (split ? sums.parts + (size_t)(tile - split_begin) * (TILE * TILE)
                                       : sums.levels + (size_t)tile * (TILE * TILE)) + off;
        unsigned long long v[FC];
#pragma unroll
        for (int c = 0; c < FC; ++c) v[c] = t[c * TILE];
        float a3[FC];
#pragma unroll
        for (int c = 0; c < FC; ++c) a3[c] = 0.f;
        if (NA > 3) {  // the parts in their order
            const float* sh = sums.shared + (size_t)(split ? split_begin + (tile - split_begin) * ways : tile) * (TILE * TILE) + off;
#pragma unroll
            for (int c = 0; c < FC; ++c) a3[c] = sh[c * TILE];
            for (int q = 1; q < (split ? ways : 1); ++q) {
                sh += TILE * TILE;
#pragma unroll
                for (int c = 0; c < FC; ++c) a3[c] += sh[c * TILE];
            }
        }
        uint2 ep[S];
        if (use_E) {
            const __nv_bfloat16* e = P.A + (size_t)i * two_np + J * 64 + FC * w;
#pragma unroll
            for (int p = 0; p < S; ++p) ep[p] = *(const uint2*)(e + (size_t)(p >> 1) * pair_stride + ((p & 1) << 5));
        }
        if (split) {
#pragma unroll
            for (int c = 0; c < FC; ++c) t[c * TILE] = 0ull;
        }
        df z[FC];
        float sd = 0.f, sf = 0.f;
#pragma unroll
        for (int c = 0; c < FC; ++c) {
            const int j = j0 + c;
            // level 2, then levels 0 and 1 as the exact pair that two_sum makes
            const int l2 = (int)(unsigned int)v[c], l01 = (int)(unsigned int)(v[c] >> 32) - (l2 >> 31);
            const float h01 = __int2float_rn(l01);
            df Pv = {h01 * (1.f / 128.f), __int2float_rn(l01 - __float2int_rn(h01)) * (1.f / 128.f)};
            if (NA > 2) Pv = df_add_f(Pv, __int2float_rn(l2) * (1.f / 16384.f));
            if (NA > 3) Pv = df_add_f(Pv, a3[c]);
            Pv = df_scale(Pv, P.scale_in_h);
            if (bad) Pv = {__int_as_float(0x7fffffff), 0.f};
            df E = {0.f, 0.f};
            if (use_E) {
                float eh = 0.f, el = 0.f;  // exact two-float sum of the digits
#pragma unroll
                for (int p = 0; p < S; ++p) {
                    const uint32_t u = (c & 2) ? ep[p].y : ep[p].x;
                    const float d = __uint_as_float((c & 1) ? (u & 0xffff0000u) : (u << 16));
                    if (p < 3)
                        eh += d;
                    else
                        el += d;
                }
                E = df_scale(fast_two_sum(eh, el), P.e_scale);
            }
            df Y = df_mul(cP, Pv);
            if (use_E) Y = df_add(Y, df_mul(cE, E));
            if (diag && i == j) Y = df_add(Y, cI);
            df O = Y;
            if (affine) {
                O = df_mul(P.dY, Y);
                if (diag && i == j) O = df_add(O, P.dI);
            }
            const bool valid = i < n && j < n;
            if (!valid) O = {0.f, 0.f};
            if (want_red && valid && i <= j) {
                const float wt = (i == j) ? 1.f : 2.f;
                if (diag && i == j) s_tr = add_df(s_tr, Y);
                const float dE = (E.h - Pv.h) + (E.l - Pv.l);
                sd += wt * dE * dE;
                sf += wt * Y.h * Y.h;
            }
            z[c] = O;
        }
        s_idem += sd;
        s_fro += sf;
        if (out64) {
#pragma unroll
            for (int c = 0; c < FC; ++c) {
                const int j = j0 + c;
                if (i < n && j < n && i <= j) {
                    const double o = add_df(0.0, z[c]);
                    out64[(size_t)i * n + j] = o;
                    if (i != j) out64[(size_t)j * n + i] = o;
                }
            }
        }
#pragma unroll
        for (int c = 0; c < FC; ++c) z[c] = df_scale(z[c], P.out_digit_scale);
        if (outp) {
            float plane_scale = 1.f;
            const float rs = P.out_rscale, rinv = 1.f / P.out_rscale;
            for (int p = 0; p < s_out; ++p) {
                unsigned short d[FC];
#pragma unroll
                for (int c = 0; c < FC; ++c) {
                    const float x = round_digit(z[c].h);
                    z[c] = df_scale(fast_two_sum(__fsub_rn(z[c].h, x), z[c].l), rs);
                    d[c] = __bfloat16_as_ushort(digit_to_bf16(x * plane_scale));
                }
                plane_scale *= rinv;
                if (diag) {
#pragma unroll
                    for (int c = 0; c < FC; ++c)
                        if (i <= j0 + c) {
                            mir[p][lane][FC * w + c] = d[c];
                            mir[p][FC * w + c][lane] = d[c];
                        }
                } else {
                    *(uint2*)&dir[p][lane][FC * w] =
                        make_uint2((uint32_t)d[0] | (uint32_t)d[1] << 16, (uint32_t)d[2] | (uint32_t)d[3] << 16);
#pragma unroll
                    for (int c = 0; c < FC; ++c) mir[p][FC * w + c][lane] = d[c];
                }
            }
            __syncthreads();
            // a plane row of 32 columns: four 16-byte pieces
            for (int q = threadIdx.x; q < s_out * 128; q += 256) {
                const int p = q >> 7, r = (q >> 2) & 31, g = q & 3;
                __nv_bfloat16* const o = outp + (size_t)(p >> 1) * pair_stride + ((p & 1) << 5) + 8 * g;
                *(uint4*)(o + (size_t)(J * 32 + r) * two_np + I * 64) = *(const uint4*)&mir[p][r][8 * g];
                if (!diag) *(uint4*)(o + (size_t)(I * 32 + r) * two_np + J * 64) = *(const uint4*)&dir[p][r][8 * g];
            }
            __syncthreads();
        }
    }
    if (!want_red) return;
    s_idem = warp_sum_f(s_idem);
    s_fro = warp_sum_f(s_fro);
    if (__any_sync(0xffffffffu, s_tr != 0.0)) {  // (NaN counts)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s_tr += __shfl_xor_sync(0xffffffffu, s_tr, o);
        if (lane == 0) atomicAdd(&P.red[0], s_tr);
    }
    if (lane == 0) {
        rsum[0][w] = s_idem;
        rsum[1][w] = s_fro;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        float x = 0.f;
        for (int q = 0; q < 8; ++q) x += rsum[threadIdx.x][q];
        atomicAdd(&P.red[1 + threadIdx.x], (double)x);
    }
}

template <int S>
int prepare_fixed() {
    PURIFY_CUDA_TRY(cudaFuncSetAttribute((const void*)digit_fixed_kernel<S>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, fixed_smem<S>()));
    cudaFuncAttributes at;  // (loads the kernel: not during a capture)
    PURIFY_CUDA_TRY(cudaFuncGetAttributes(&at, (const void*)digit_finish_kernel<S>));
    return PURIFY_OK;
}

template <int S>
int launch_fixed(const DigitStep& st, cudaStream_t stream) {
    FixedLaunch L;
    PURIFY_TRY(fill_digit_params(st, &L.prm, &L.map_a, &L.map_b));
    const int T = st.n_pad / TILE, tiles = T * (T + 1) / 2;
    L.sums = *st.fixed;
    L.err = st.err;
    L.wait_cycles = st.wait_cycles;
    digit_step_split(st, tiles, &L.split_begin, &L.ways);
    L.items = L.split_begin + (tiles - L.split_begin) * L.ways;
    // An item's halves on two CTAs while each gets one (the accumulators are
    // independent, so their sums keep their order). Per product, whole items ->
    // halves: n = 200 (6 items) 19.6 -> 17 us, n = 512 (40) 21.2 -> 19.0 us. With
    // more items than half the CTAs it does not pay: half 0 takes in as many
    // operand bytes for fewer MMAs (n = 1500, 78 items: 78 -> 91 us).
    L.halves = S > NUM_ACC - 1 && 2 * L.items <= st.max_ctas ? 2 : 1;
    const int grid = std::min(L.items * L.halves, st.max_ctas);
    PURIFY_TRY(prepare_digit_fixed());
    PURIFY_CUDA_TRY(launch_chained(digit_fixed_kernel<S>, (unsigned)grid, (unsigned)kThreads, fixed_smem<S>(), stream, L));
    const int nb = st.n_pad / 32, blocks = nb * (nb + 1) / 2;
    PURIFY_CUDA_TRY(launch_chained(digit_finish_kernel<S>, (unsigned)std::min(blocks, st.max_ctas * 4), 256u, 0, stream, L.prm,
                                   L.sums, L.split_begin, L.ways, blocks));
    count_launches(2);
    return PURIFY_OK;
}

}  // namespace

int prepare_digit_fixed() {
    static std::mutex mu;
    static bool done = false;
    std::lock_guard<std::mutex> g(mu);
    if (done) return PURIFY_OK;
    PURIFY_TRY(prepare_fixed<2>());
    PURIFY_TRY(prepare_fixed<3>());
    PURIFY_TRY(prepare_fixed<4>());
    PURIFY_TRY(prepare_fixed<5>());
    PURIFY_TRY(prepare_fixed<6>());
    done = true;
    return PURIFY_OK;
}

bool digits_fixed_size(int n_pad, int ctas) {
    const int T = n_pad / TILE;
    return T * (T + 1) / 2 < 2 * ctas;
}

bool digits_fixed_wanted(const DigitStep& st) {
    if (!st.fixed || !st.err || st.max_ctas < 1 || st.kc_cnt || st.bnorm2 || st.a_idx) return false;
    if (st.rbits != 7 || st.s_in < 2 || st.s_in > kMaxDigitPlanes) return false;
    const int T = st.n_pad / TILE;
    return digits_fixed_size(st.n_pad, st.max_ctas) && T * (T + 1) / 2 <= st.fixed->tiles;
}

// A tile has at most four parts; a product has less than two waves of tiles and at
// most a wave of parts, two or more to a split tile (digit_split_plan).
int alloc_fixed_sums(int tiles, int ctas, FixedSums* f) {
    const size_t tile = (size_t)TILE * TILE;
    f->parts_bytes = std::min(tiles, ctas / 2 + 1) * tile * sizeof(unsigned long long);
    PURIFY_CUDA_TRY(cudaMalloc(&f->levels, tiles * tile * sizeof(unsigned long long)));
    PURIFY_CUDA_TRY(cudaMalloc(&f->parts, f->parts_bytes));
    PURIFY_CUDA_TRY(cudaMalloc(&f->shared, std::min(4 * tiles, 2 * ctas) * tile * sizeof(float)));
    f->tiles = tiles;
    return PURIFY_OK;
}
void free_fixed_sums(FixedSums* f) {
    cudaFree(f->levels);
    cudaFree(f->parts);
    cudaFree(f->shared);
    *f = FixedSums();
}

int launch_digit_fixed(const DigitStep& st, cudaStream_t stream) {
    switch (st.s_in) {
        case 2: return launch_fixed<2>(st, stream);
        case 3: return launch_fixed<3>(st, stream);
        case 4: return launch_fixed<4>(st, stream);
        case 5: return launch_fixed<5>(st, stream);
        case 6: return launch_fixed<6>(st, stream);
        default: return PURIFY_ERR_INVALID_ARG;
    }
}

}  // namespace purify
