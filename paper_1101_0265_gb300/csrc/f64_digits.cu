// Float64 symmetric steps on the tcgen05 tensor cores.
//
// GB300's float64 pipe runs 2 FMAs per clock and SM (1.26 TFLOP/s on the
// chip), so a float64 product there is bound by that pipe at any size.  Here
// the product is taken on the bf16 tensor pipe (1.9 PFLOP/s measured) with
// float64's accuracy relative to the rows' norms: the operands are cut into
// integer digits whose products and leading sums are exact in the fp32
// accumulators, and the sums are put together in 64-bit integers (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012), with
// digits of 7 bits).
//
// Digits.  Row i of a symmetric operand has the exponent e_i with
// ||x_i||_2 <= 2^e_i (and > 2^(e_i - 2)); x_ij = 2^(e_i - 8) sum_p d_p 2^(-7p)
// with |d_0| <= 256 and |d_p| <= 64 for p = 1..7: 57 bits below 2^e_i, an
// entry's error is at most 2^(e_i - 58).  Digit p is stored as the bf16 value
// d_p 2^(-7p), exactly.
//
// Product.  P_ij = 2^(e_i + e_j - 16) sum_l 2^(-7l) L_l with the level sums
// L_l = sum_{p + q = l} sum_k d_p(i, k) d_q(j, k), l = 0..8 (p, q <= 7): 43
// digit pairs.  What is left out (levels >= 9 and the digits' own rounding) is
// about 2^-57 of ||x_i|| ||x_j|| (at worst 4 sqrt(n) times that), for dense rows
// below the rounding of a chain of n float64 FMAs.  (With level 8 cut to its middle
// pair, 37 pairs, off-diagonal entries came out 2.5 times further off than with
// FMAs at n = 4096.)  A level sum over at most 1024 columns stays below 2^24 for l
// <= 4 whatever the digits are (Cauchy-Schwarz for the pairs with d_0, at most 3 x
// 1024 x 2^12 for the others) and is then exact in fp32; level 5 may exceed it by a
// sixteenth in the worst case, at 2^-51 of the leading term per unit, and levels 6
// to 8 are rounded in fp32 (7 and 8 once more, to 32 of level 7's units, when they
// are emptied).  So an accumulator is emptied at least every 1024 columns, as an
// integer: each segment adds its levels, shifted into units of 2^(e_i + e_j - 60),
// to a 64-bit integer per element (|P_ij| <= 2^(e_i + e_j): the sum fits).
// Integer sums do not depend on their order, so the result is the same on every
// run; with another number of SMs the segments are cut elsewhere and the last
// bits, from level 5 on, may differ.
//
// Work.  Eight 128 x 128 accumulators would need twice the 512 columns of
// tensor memory, so a tile's range is done in two passes: levels 0..3 from
// digits 0..3 (10 digit pairs), then levels 4..8 from all digits (33; levels 7
// and 8 share an accumulator).
// Whole waves of tiles go round-robin, so that the CTAs walk k together and
// share panels in L2; the tiles of the last, partial wave are cut evenly over
// the grid at stage boundaries (at n = 256, three tiles on 72 of 103 CTAs).
//
// Measured, one step (float64 FMA kernel -> here): n = 256 23 -> 19 us, n = 1000
// 896 -> 57 us, n = 4096 56 ms -> 1.69 ms, of which the product kernel is about 1.5
// ms: 2.0 PFLOP/s of digit pairs (cuBLAS bf16 burst: 1.9).  Errors of one step on
// a dense rotated matrix against extended precision at n = 4096: largest 2.2e-15
// -> 7e-17, rms 1.8e-17 -> 2.4e-18.  Matrices with entries far below their rows'
// norms are another matter: see the test of the result below.
//
// A step is three launches: split (unless the operand's digits are still at
// hand), product, finish.  An operand with an infinity, a NaN or a row scale
// above 2^400 sets flags[0]: the kernels of that step and of all later ones leave
// at once, and the caller goes on with the float64 FMA kernel, which carries such
// values (a run from its start, the gap estimate and the refinement from that
// step).  Rows that underflow (a decoupled unoccupied orbital squared step after
// step) keep the scale 2^-400.
#include "f64_digits.h"

#include <algorithm>
#include <type_traits>

#include "digits_kernel.cuh"
#include "tile_sums.cuh"

namespace purify {

using namespace dk;

int make_quad_map(CUtensorMap* map, const __nv_bfloat16* planes, int n_pad);  // digits_tc.cu

namespace {

constexpr int kDigits = 8;
constexpr int kStages = 3;
constexpr int kStageBytes = 64 * 1024;
constexpr int kBoxBytes = TILE * 128;  // 128 rows of four planes' 16-wide k-chunks
// 16 epilogue warps, each 32 rows x 32 columns of a tile: with 8 an emptying of the
// accumulators waits on its own arithmetic (two warps per scheduler)
constexpr int kEpi = 16;
constexpr int kThreads = 64 + 32 * kEpi;
constexpr int kMaxRegs = 96;  // 18 warps: five on a sub-partition of 16384 registers
constexpr int kExpLimit = 400;
// MMAs per stage, which also measure the work: a high stage is 32 columns of
// levels 0..3, a low stage 16 columns of levels 4..8
constexpr int kHiCost = 20, kLoCost = 33;
constexpr int kRange32 = 32;  // 1024 columns between two emptyings, in 32-column chunks
constexpr int kCost32 = kHiCost + 2 * kLoCost;
constexpr int kRangeCost = kRange32 * kCost32;
// A CTA's share of the last wave is at least this: one high stage, so that in small
// products no CTA empties its accumulators twice. (A low stage costs 33, so some
// shares hold the start of no stage: 31 of 103 at n = 256.) n = 256, per step: 20.5
// us with 20, 24.6 with 30, 25.0 with 60; from n = 333 on the grid is full and it
// does not matter.
constexpr int kMinCost = 20;
constexpr int ERR_F64_WAIT = 32;
constexpr int kSmemBytes = 1024 + kStages * kStageBytes + 256;
// From n = 160 a step here is faster than the float64 FMA kernel's (n = 130 17.7
// against 16.3 us a step, n = 160 18.1 against 18.2, n = 192 18.4 against 20.6, n = 257
// 25 against 41); the largest size bounds the buffers (39 GB).
constexpr int64_t kF64DigitsMinN = 160, kF64DigitsMaxN = 1 << 15;

struct F64Product {
    CUtensorMap map_a, map_b;
    unsigned long long* T;
    int* flags;
    long long wait_cycles;            // bound of one work wait
    int tiles_per_row, tiles, whole;  // whole: full waves of tiles
};

// The segments of one CTA, the same sequence in every role: a tile, a pass and
// a run of stages.
struct Segment {
    int ti, tj, lo, k0, count;  // k0 in 32- (high) or 16-column (low) chunks
};

struct Walk {
    int T, nk32, whole, grid, tile_cost;
    int w = -1, tile = 0, pos = 0, end = 0;
    long long tb, te;
    __device__ explicit Walk(const F64Product& L) {
        T = L.tiles_per_row;
        nk32 = T * 4;
        whole = L.whole;
        grid = gridDim.x;
        tile_cost = nk32 * kCost32;
        const long long total = (long long)(L.tiles - whole * grid) * tile_cost;
        tb = total * blockIdx.x / grid;
        te = total * (blockIdx.x + 1) / grid;
    }
    __device__ bool next(Segment& g) {
        for (;;) {
            if (pos >= end) {
                ++w;
                if (w < whole) {
                    tile = blockIdx.x + w * grid;
                    pos = 0;
                    end = tile_cost;
                } else {
                    if (tb >= te) return false;
                    const int q = (int)(tb / tile_cost);
                    tile = whole * grid + q;
                    pos = (int)(tb - (long long)q * tile_cost);
                    end = (int)min((long long)tile_cost, pos + (te - tb));
                    tb += end - pos;
                }
            }
            // the stages that start inside [pos, end) of this range's pass
            const int r = pos / kRangeCost, base = r * kRangeCost;
            const int kr = min(kRange32, nk32 - r * kRange32);
            const int hc = kHiCost * kr, off = pos - base;
            const int e = min(end - base, kCost32 * kr);
            int s0, s1;
            if (off < hc) {
                const int eh = min(e, hc);
                s0 = (off + kHiCost - 1) / kHiCost;
                s1 = (eh + kHiCost - 1) / kHiCost;
                g.lo = 0;
                g.k0 = r * kRange32 + s0;
                pos = base + eh;
            } else {
                s0 = (off - hc + kLoCost - 1) / kLoCost;
                s1 = (e - hc + kLoCost - 1) / kLoCost;
                g.lo = 1;
                g.k0 = 2 * r * kRange32 + s0;
                pos = base + e;
            }
            if (s1 > s0) {
                g.count = s1 - s0;
                decode_banded(tile, T, g.ti, g.tj);
                return true;
            }
        }
    }
};

// Descriptor offset (16-byte units) of digit plane p inside an operand's
// 16-column chunk: four planes side by side in a 128-byte row.
__host__ __device__ constexpr int quad_off(int p) { return ((p >> 2) * kBoxBytes + (p & 3) * 32) >> 4; }

// Stage layout: A at 0, B at 32 KB.  High: two 16-column chunks of planes
// 0..3 each; low: one chunk of planes 0..3 and 4..7.
__device__ __forceinline__ void issue_high(uint32_t tmem, uint64_t da, uint64_t db, uint32_t later) {
#pragma unroll
    for (int kk = 0; kk < 2; ++kk)
#pragma unroll
        for (int l = 0; l < 4; ++l)
#pragma unroll
            for (int p = 0; p <= l; ++p)
                mma_bf16(tmem + (uint32_t)(l * TILE), da + (uint64_t)(kk * (kBoxBytes >> 4) + quad_off(p)),
                         db + (uint64_t)(kk * (kBoxBytes >> 4) + quad_off(l - p)), IDESC,
                         (kk > 0 || p > 0) ? 1u : later);
}

__device__ __forceinline__ void issue_low(uint32_t tmem, uint64_t da, uint64_t db, uint32_t later) {
#pragma unroll
    for (int l = 4; l < 8; ++l)
#pragma unroll
        for (int p = 0; p <= l; ++p)
            mma_bf16(tmem + (uint32_t)((l - 4) * TILE), da + (uint64_t)quad_off(p), db + (uint64_t)quad_off(l - p),
                     IDESC, p > 0 ? 1u : later);
#pragma unroll
    for (int p = 1; p < 8; ++p)
        mma_bf16(tmem + (uint32_t)(3 * TILE), da + (uint64_t)quad_off(p), db + (uint64_t)quad_off(8 - p), IDESC, 1u);
}

// The four accumulators of one element as a 64-bit integer in units of
// 2^-60, modulo 2^64: 32-bit halves (64-bit integer operations run on the
// float64 pipe).  Conversions of floats to integers run at 16 per clock and SM,
// four per element would take 4096 cycles of an emptying; levels that stay below
// 2^22 (0 and 1: |L_1| <= 2 x 2^8 x 64 x 32; 7 in units of 32) are read off the
// bits of a sum with 1.5 2^23 instead, and one of the larger low levels in two
// such pieces.
__device__ __forceinline__ uint2 levels_high(float a0, float a1, float a2, float a3) {
    const unsigned int l0 = __float_as_uint(a0 + kMagic), l1 = __float_as_uint(fmaf(a1, 128.f, kMagic));
    const int l2 = __float2int_rn(a2 * 16384.f), l3 = __float2int_rn(a3 * 2097152.f);
    // (l0 << 44) + (l1 << 37) + (l2 << 30) + (l3 << 23); the magic bits shifted
    // into the high half go off again
    const unsigned int x = (unsigned int)l2 << 30, lo = x + ((unsigned int)l3 << 23);
    const unsigned int hi = (l0 << 12) + (l1 << 5) + (unsigned int)(l2 >> 2) + (unsigned int)(l3 >> 9) +
                            (lo < x ? 1u : 0u) - ((kMagicBits << 12) + (kMagicBits << 5));
    return make_uint2(lo, hi);
}

__device__ __forceinline__ uint2 levels_low(float a4, float a5, float a6, float a7) {
    const int l4 = __float2int_rn(a4 * 268435456.f), l5 = __float2int_rn(a5 * 34359738368.f);
    // level 6 = 4096 t + r, and level 7 (with 8) / 32
    const float v6 = a6 * 4398046511104.f;
    const float t = fmaf(v6, 1.f / 4096.f, kMagic);
    const float r = fmaf(t - kMagic, -4096.f, v6) + kMagic;
    const int z = (int)((__float_as_uint(t) - kMagicBits) << 14) + (int)((__float_as_uint(r) - kMagicBits) << 2) +
                  (int)(__float_as_uint(fmaf(a7, 17592186044416.f, kMagic)) - kMagicBits);
    // (l4 << 16) + (l5 << 9) + z
    const unsigned int x = (unsigned int)l4 << 16, s = x + ((unsigned int)l5 << 9), lo = s + (unsigned int)z;
    const unsigned int hi = (unsigned int)(l4 >> 16) + (unsigned int)(l5 >> 23) + (unsigned int)(z >> 31) +
                            (s < x ? 1u : 0u) + (lo < s ? 1u : 0u);
    return make_uint2(lo, hi);
}

__global__ void __maxnreg__(kMaxRegs) f64_digit_product_kernel(const __grid_constant__ F64Product L) {
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

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * kStages; ++i) mbar_init(smem_u32(&full_bar[i]), 1);
        mbar_init(smem_u32(tmem_full), 1);
        mbar_init(smem_u32(tmem_empty), kEpi);
        mbar_init(smem_u32(drain), 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), 4 * TILE);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    Walk walk(L);
    Segment g;
    grid_dependency_wait();
    // a step that is not taken (written by earlier kernels only: uniform over the grid)
    const bool skip = L.flags[0] != 0;

    if (skip) {
    } else if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            while (ok && walk.next(g)) {
                for (int c = 0; c < g.count; ++c, ++it) {
                    const int st = it % kStages;
                    if ((it >= kStages &&
                         !mbar_wait_for(smem_u32(&empty_bar[st]), (uint32_t)(((it / kStages) & 1) ^ 1), L.wait_cycles)) ||
                        *abort_flag) {
                        ok = false;
                        break;
                    }
                    const uint32_t fb = smem_u32(&full_bar[st]);
                    const uint32_t sa = smem_u32(base + (size_t)st * kStageBytes);
                    const uint32_t sb = sa + 2 * kBoxBytes;
                    mbar_arrive_expect_tx(fb, (uint32_t)kStageBytes);
                    // high: two chunks of planes 0..3; low: one chunk of each four
                    const int x0 = (g.k0 + c) * (g.lo ? 64 : 128), x1 = g.lo ? x0 : x0 + 64;
                    tma_load_3d(sa, &L.map_a, fb, x0, g.ti * TILE, 0);
                    tma_load_3d(sb, &L.map_b, fb, x0, g.tj * TILE, 0);
                    tma_load_3d(sa + kBoxBytes, &L.map_a, fb, x1, g.ti * TILE, g.lo);
                    tma_load_3d(sb + kBoxBytes, &L.map_b, fb, x1, g.tj * TILE, g.lo);
                }
            }
            if (!ok) {
                atomicOr(L.flags + 1, ERR_F64_WAIT);
                *abort_flag = 1;
            }
            // wait (bounded) for the copies still in flight
            for (int k = (it > kStages ? it - kStages : 0); k < it; ++k)
                mbar_wait_for(smem_u32(&full_bar[k % kStages]), (uint32_t)((k / kStages) & 1));
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint64_t desc_base = smem_desc(smem_u32(base));
            int it = 0, lt = 0;
            bool ok = true;
            for (; ok && walk.next(g); ++lt) {
                if (lt > 0 && !mbar_wait_for(smem_u32(tmem_empty), (uint32_t)((lt - 1) & 1), L.wait_cycles)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                for (int c = 0; c < g.count; ++c, ++it) {
                    const int st = it % kStages;
                    if (!mbar_wait_for(smem_u32(&full_bar[st]), (uint32_t)((it / kStages) & 1), L.wait_cycles)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t da = desc_base + (uint64_t)((st * kStageBytes) >> 4);
                    const uint64_t db = da + (uint64_t)((2 * kBoxBytes) >> 4);
                    if (g.lo)
                        issue_low(tmem, da, db, c > 0 ? 1u : 0u);
                    else
                        issue_high(tmem, da, db, c > 0 ? 1u : 0u);
                    mma_commit(smem_u32(&empty_bar[st]));
                }
                if (ok) mma_commit(smem_u32(tmem_full));
            }
            if (!ok) {
                atomicOr(L.flags + 1, ERR_F64_WAIT);
                *abort_flag = 1;
            }
            mma_commit(smem_u32(drain));
            mbar_wait_for(smem_u32(drain), 0);
        }
    } else {
        // epilogue warps: lane quarter warp % 4, the (warp - 2) / 4-th 32 columns
        const int quarter = warp & 3, col0 = ((warp - 2) >> 2) * (TILE * 4 / kEpi);
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)col0;
        for (int lt = 0; walk.next(g); ++lt) {
            bool ready = mbar_wait_for(smem_u32(tmem_full), (uint32_t)(lt & 1), L.wait_cycles);
            if (!ready) {
                atomicOr(L.flags + 1, ERR_F64_WAIT);
                *abort_flag = 1;
            }
            ready = __all_sync(0xffffffffu, ready && !*abort_flag);  // tcgen05.ld is warp-collective
            if (!ready) break;
            tc_fence_after();
            // column-major inside a tile: a warp adds 32 consecutive integers
            unsigned long long* t = L.T + (size_t)(g.tj * (g.tj + 1) / 2 + g.ti) * (TILE * TILE) + quarter * 32 + lane +
                                    col0 * TILE;
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
                if (g.ti == g.tj && quarter > ((col0 + 8 * q) >> 5)) continue;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float a0 = __uint_as_float(v[c]), a1 = __uint_as_float(v[8 + c]),
                                a2 = __uint_as_float(v[16 + c]), a3 = __uint_as_float(v[24 + c]);
                    const uint2 u = g.lo ? levels_low(a0, a1, a2, a3) : levels_high(a0, a1, a2, a3);
                    atomicAdd(t + (8 * q + c) * TILE, (unsigned long long)u.y << 32 | u.x);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 4 * TILE);
    }
}

// ---- split: float64 rows -> exponents and digit planes ------------------------

// Element offset of (plane p, row i, column j): planes 4m..4m+3 side by side
// in 16-column chunks, 128-byte rows.
__device__ __forceinline__ size_t quad_index(int p, int i, int j, int n_pad) {
    return (size_t)(p >> 2) * 4 * n_pad * n_pad + (size_t)i * 4 * n_pad + ((j >> 4) << 6) + ((p & 3) << 4) + (j & 15);
}

template <int TPR, typename V, typename Op>
__device__ __forceinline__ V row_reduce(V v, Op op) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    if constexpr (TPR > 32) {
        __shared__ V part[TPR / 32];
        __syncthreads();
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
        __syncthreads();
        v = part[0];
#pragma unroll
        for (int w = 1; w < TPR / 32; ++w) v = op(v, part[w]);
    }
    return v;
}

// TPR threads per row (a warp for short rows, the block of 256 for long ones),
// NG groups of four consecutive columns per thread, held in registers between
// the three passes over the row (largest exponent, 2-norm, digits); NG = 0:
// longer rows, read again from L1 / L2 by each pass.  Bound by HBM for large n (8
// bytes read and 16 written per element), by load latency for small n.
// Integer arithmetic and float32 only.
template <int TPR, int NG>
__global__ void __launch_bounds__(256)
f64_split_kernel(const double* __restrict__ X, int n, int n_pad, __nv_bfloat16* __restrict__ planes,
                 int* __restrict__ exps, int* flags, int step) {
    grid_dependency_wait();
    // (a block of this launch may set it: decide once per block)
    if (__syncthreads_or(*(volatile int*)flags != 0)) return;
    const int i = (int)blockIdx.x * (256 / TPR) + (int)threadIdx.x / TPR;  // < n_pad, a multiple of 128
    const int t = threadIdx.x % TPR;
    const double* row = X + (size_t)i * n;
    const bool in = i < n, vec = (n & 1) == 0;
    auto load4 = [&](int j0, double (&x)[4]) {
        x[0] = x[1] = x[2] = x[3] = 0.0;
        if (!in) return;
        if (vec && j0 + 3 < n) {
            const double2 u = *(const double2*)(row + j0), v = *(const double2*)(row + j0 + 2);
            x[0] = u.x;
            x[1] = u.y;
            x[2] = v.x;
            x[3] = v.y;
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (j0 + c < n) x[c] = row[j0 + c];
        }
    };
    double held[NG > 0 ? NG : 1][4];
    if constexpr (NG > 0) {
#pragma unroll
        for (int g = 0; g < NG; ++g) load4(4 * (t + g * TPR), held[g]);
    }
    auto for_row = [&](int end, auto&& body) {
        if constexpr (NG > 0) {
#pragma unroll
            for (int g = 0; g < NG; ++g)
                if (4 * (t + g * TPR) < end) body(4 * (t + g * TPR), held[g]);
        } else {
            for (int j0 = 4 * t; j0 < end; j0 += 4 * TPR) {
                load4(j0, held[0]);
                body(j0, held[0]);
            }
        }
    };
    unsigned int top = 0;  // the largest high word: sign off, exponent and 20 leading bits
    for_row(n, [&](int, double (&x)[4]) {
#pragma unroll
        for (int c = 0; c < 4; ++c) top = max(top, (unsigned int)__double2hiint(x[c]) & 0x7fffffffu);
    });
    top = row_reduce<TPR>(top, [](unsigned int a, unsigned int b) { return max(a, b); });
    const int emax = (int)(top >> 20);
    // sum of squares relative to 2^(emax - 1023), from the high words
    float ss = 0.f;
    for_row(n, [&](int, double (&x)[4]) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const unsigned int h = (unsigned int)__double2hiint(x[c]) & 0x7fffffffu;
            const int d = (int)(h >> 20) - emax;
            const float m = d > -60 ? __uint_as_float((unsigned int)(127 + d) << 23 | (h & 0xfffffu) << 3) : 0.f;
            ss = fmaf(m, m, ss);
        }
    });
    ss = row_reduce<TPR>(ss, [](float a, float b) { return a + b; });
    // the smallest k with 4^k > ss (raised by the truncation and the sum's rounding)
    const int lg = (int)(__float_as_uint(ss * 1.01f) >> 23) - 127;
    // a row of zeros or below 2^-400 keeps the exponent -400: what its digits leave
    // out is below 2^-457
    const int e = max(emax == 0 ? -kExpLimit : emax - 1023 + ((lg + 2) >> 1), -kExpLimit);
    if (t == 0) {
        if (emax == 2047 || e > kExpLimit) atomicCAS(flags, 0, step + 1);  // digits cannot hold it
        exps[i] = e;
    }
    for_row(n_pad, [&](int j0, double (&x)[4]) {
        uint32_t w[kDigits][2];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            // x 2^(57 - e), rounded to an integer of at most 58 bits
            const unsigned int h = (unsigned int)__double2hiint(x[c]), l = (unsigned int)__double2loint(x[c]);
            const int E = (int)((h >> 20) & 0x7ffu);
            unsigned long long m = (unsigned long long)((h & 0xfffffu) | 0x100000u) << 32 | l;
            const int sh = E - 1018 - e;  // <= 5
            if (E == 0 || sh < -54)
                m = 0;
            else if (sh >= 0)
                m <<= sh & 7;
            else
                m = (m + (1ull << (-sh - 1))) >> -sh;
            long long f = (h >> 31) ? -(long long)m : (long long)m;
            // balanced digits from the last one up: |d_p| <= 64
            int d[kDigits];
#pragma unroll
            for (int p = kDigits - 1; p > 3; --p) {
                f += 64;
                d[p] = (int)((unsigned int)f & 127u) - 64;
                f >>= 7;
            }
            int f32 = (int)f;
#pragma unroll
            for (int p = 3; p > 0; --p) {
                f32 += 64;
                d[p] = (f32 & 127) - 64;
                f32 >>= 7;
            }
            d[0] = f32;
            float scale = 1.f;
#pragma unroll
            for (int p = 0; p < kDigits; ++p) {
                // d_p as a float by its bits (|d_p| <= 256), then its true scale; bf16 holds it exactly
                const float v = (__int_as_float(0x4B400000 + d[p]) - 12582912.f) * scale;
                const uint32_t b = __float_as_uint(v) >> 16;
                if (c & 1)
                    w[p][c >> 1] |= b << 16;
                else
                    w[p][c >> 1] = b;
                scale *= 1.f / 128.f;
            }
        }
#pragma unroll
        for (int p = 0; p < kDigits; ++p)
            *(uint2*)(planes + quad_index(p, i, j0, n_pad)) = make_uint2(w[p][0], w[p][1]);
    });
}

// ---- finish: fixed-point product -> the step's polynomial ----------------------

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// v 2^ex, rounded to nearest even (|ex| < 900, |v| < 2^63): integer operations
// on 32-bit halves, where a conversion and a multiplication would take the
// float64 pipe.
__device__ __forceinline__ double fixed_to_double(uint2 v, int ex) {
    const unsigned int sign = v.y & 0x80000000u;
    unsigned int lo = v.x, hi = v.y;
    if (sign) {
        lo = 0u - lo;
        hi = ~hi + (lo == 0u ? 1u : 0u);
    }
    if ((lo | hi) == 0u) return 0.0;
    const int z = hi ? __clz(hi) : 32 + __clz(lo);
    if (z >= 32) {
        hi = lo;
        lo = 0u;
    }
    hi = __funnelshift_l(lo, hi, z);  // (shifts by z mod 32)
    lo <<= z & 31;
    // bit 63 leads: 53 bits kept, ties to even
    const unsigned int rem = lo & 0x7ffu, mlo = hi << 21 | lo >> 11;
    const unsigned int inc = (rem > 0x400u || (rem == 0x400u && (mlo & 1u))) ? 1u : 0u;
    const unsigned int rlo = mlo + inc;
    const unsigned int rhi = (hi >> 11) + (rlo < inc ? 1u : 0u) + ((unsigned int)(63 - z + ex + 1022) << 20);
    return __hiloint2double((int)(sign | rhi), (int)rlo);
}

// One pass of a finish block over 32 rows (lane: i = i0 + tx) x 8 NQ columns from
// j0 of the 32 x 32 block (I, J); DIAG: I = J.  The diagonal's extra terms are
// kept out of the other blocks' code: an instruction whose predicate is off
// still takes its turn on the float64 pipe.
template <int NQ, bool HAS_E, bool AFFINE, bool DIAG>
__device__ __forceinline__ void finish_pass(const uint2 (&v)[NQ], const double (&e)[NQ], const int (&ex)[NQ], int i,
                                            int j0, int n, double* __restrict__ C, double cP, double cE, double cI,
                                            double dY, double dI, double (*tile)[33], double& s_tr, double& s_idem) {
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    double sd = 0.0;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int c = ty + 8 * q, j = j0 + c;
        double out = 0.0;
        if (i < n && j < n && (!DIAG || i <= j)) {
            const double p = fixed_to_double(v[q], ex[q]);
            double y = cP * p;
            if (HAS_E) {
                y = fma(cE, e[q], y);
                const double d = e[q] - p;
                sd = fma((DIAG && i == j) ? 0.5 * d : d, d, sd);
            }
            if (DIAG && i == j) y += cI;
            out = y;
            if (AFFINE) out = dY * y;
            if (DIAG && i == j) {
                out += dI;
                s_tr += y;
            }
            C[(size_t)j * n + i] = out;
        }
        tile[c][tx] = out;
    }
    if (HAS_E) s_idem += sd;  // half of the sum over the whole matrix
}

// Y = cP P + cE E + cI I, C = dY Y + dI I (with mirror) over pieces of the 32 x
// 32 blocks I <= J: 32 rows x 8 NQ columns per pass of a block of threads.
// red[0] += trace(Y), red[1] += ||E - P||_F^2 (HAS_E).  Reads each fixed-point
// entry once and clears it for the next step.  At most four float64
// operations per element of the upper triangle: at n = 4096 they take 60 us of
// that pipe, the 40 bytes per upper element 50 us of HBM; 85 us measured (185
// without reading a piece ahead, 372 with conversions and the diagonal's terms on
// the float64 pipe as well).  NQ = 1
// spreads small matrices over more SMs (n = 256: 36 blocks of 32 x 32).
template <int NQ, bool HAS_E, bool AFFINE>
__global__ void __launch_bounds__(256, 4)
f64_finish_kernel(uint2* __restrict__ T, const int* __restrict__ ea, const int* __restrict__ eb,
                  const double* __restrict__ E, double* __restrict__ C, int n, int pieces, double cP, double cE,
                  double cI, double dY, double dI, double* red, const int* __restrict__ flags) {
    constexpr int PB = 4 / NQ;  // pieces per 32 x 32 block
    __shared__ double tile[8 * NQ][33];
    __shared__ double rsum[256];
    grid_dependency_wait();
    if (flags[0]) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    double s_tr = 0.0, s_idem = 0.0;
    bool any_diag = false;
    // a piece's place, and its entries and E, read one piece ahead
    struct Piece {
        int I, J, c0;
        uint2* t;
        uint2 v[NQ];
        double e[NQ];
        int ex[NQ];
    } cur, nxt;
    auto fetch = [&](int u, Piece& p) {
        const int b = u / PB;
        p.c0 = (u % PB) * 8 * NQ;
        int J = (int)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
        while ((J + 1) * (J + 2) / 2 <= b) ++J;
        while (J * (J + 1) / 2 > b) --J;
        p.J = J;
        p.I = b - J * (J + 1) / 2;
        p.t = T + (size_t)((J >> 2) * ((J >> 2) + 1) / 2 + (p.I >> 2)) * (TILE * TILE) +
              (size_t)((J & 3) * 32 + p.c0) * TILE + (p.I & 3) * 32 + tx;
        const int i = p.I * 32 + tx, j0 = J * 32 + p.c0;
        const int ei = ea[i] - 60;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int c = ty + 8 * q, j = j0 + c;
            p.v[q] = __ldcs(p.t + c * TILE);
            p.e[q] = (HAS_E && i < n && j < n) ? E[(size_t)j * n + i] : 0.0;
            p.ex[q] = ei + eb[j];
        }
    };
    if ((int)blockIdx.x < pieces) fetch(blockIdx.x, nxt);
    for (int u = blockIdx.x; u < pieces; u += gridDim.x) {
        cur = nxt;
        if (u + (int)gridDim.x < pieces) fetch(u + gridDim.x, nxt);
        const int I = cur.I, J = cur.J, i = I * 32 + tx, j0 = J * 32 + cur.c0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) cur.t[(ty + 8 * q) * TILE] = make_uint2(0u, 0u);
        if (I == J) {
            any_diag = true;
            finish_pass<NQ, HAS_E, AFFINE, true>(cur.v, cur.e, cur.ex, i, j0, n, C, cP, cE, cI, dY, dI, tile, s_tr, s_idem);
        } else {
            finish_pass<NQ, HAS_E, AFFINE, false>(cur.v, cur.e, cur.ex, i, j0, n, C, cP, cE, cI, dY, dI, tile, s_tr, s_idem);
        }
        __syncthreads();
        // the row segments (i, j0 .. j0 + 8 NQ): 8 NQ threads a row
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int w = threadIdx.x + 256 * q, r = w / (8 * NQ), c = w % (8 * NQ);
            const int i2 = I * 32 + r, j2 = j0 + c;
            if (j2 < n && i2 < j2) C[(size_t)i2 * n + j2] = tile[c][r];
        }
        __syncthreads();
    }
    if (!red) return;
    // one warp adds up the block (a shuffle tree in every warp would put eight
    // times as many additions on the float64 pipe); the trace only where the
    // block met the diagonal
    auto block_total = [&](double x) -> double {
        rsum[threadIdx.x] = x;
        __syncthreads();
        double w = 0.0;
        if (ty == 0) {
#pragma unroll
            for (int q = 0; q < 8; ++q) w += rsum[tx + 32 * q];
            w = warp_sum_d(w);
        }
        __syncthreads();
        return w;
    };
    if (HAS_E) {
        const double w = block_total(s_idem);
        if (threadIdx.x == 0) atomicAdd(&red[1], 2.0 * w);
    }
    if (any_diag) {
        const double w = block_total(s_tr);
        if (threadIdx.x == 0) atomicAdd(&red[0], w);
    }
}

// ---- small entries of the result ----------------------------------------------
//
// A chain of FMAs keeps P_ij to about n 2^-53 S_ij with S_ij = sum_k |x_ik| |x_kj|;
// digits keep it to about 2^-57 ||x_i|| ||x_j||, which is no worse while S_ij >=
// ||x_i|| ||x_j|| / (16 n).  Dense densities are far above that (rotated spectra of
// fillings 0.25 to 0.7: 330 to 6800 times, n = 160 to 1000), but in a matrix that
// decays away from the diagonal, or whose parts are weakly coupled, the entries
// between distant rows are far below it (gapped alternating chain, n = 240:
// relative errors of 1e-7 at entries of 3e-12, nothing left below 1e-18).  So the
// density of a run is tested pair by pair, and a run with a pair below the bound
// is the FMA kernel's.  The iterates need no test of their own: where one of them
// has small entries and the density has none, those do not show in it beyond
// 2^-57 of the norms.
//
// Both kernels work in float32 and go to float64 only for what does not fit there;
// the conversions still fill the float64 pipe (row pass at n = 4096: 43 us, that
// pipe 90 % busy; reading D takes 20). All in float64 the test was 36 us of a call
// at n = 1000 and 230 us at n = 4096 (1.6 and 24.6 ms), now 12 and 140 us (n = 256:
// nothing that shows).

struct RowScale {
    double inv;      // 1 / ||d_i|| (0: the row is below 2^-400 and not tested)
    double diag;     // |d_ii|
    float invf, diagf;
};

// One warp per row.
__global__ void __launch_bounds__(256)
f64_row_scale_kernel(const double* __restrict__ D, int n, RowScale* __restrict__ rows, const int* __restrict__ flags) {
    grid_dependency_wait();
    if (flags[0]) return;
    const int i = (int)blockIdx.x * 8 + (int)threadIdx.x / 32, lane = threadIdx.x & 31;
    if (i >= n) return;
    const double* row = D + (size_t)i * n;
    float sf = 0.f;
    for (int c0 = 0; c0 < n; c0 += 256) {
        float x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = c0 + 32 * q + lane < n ? (float)row[c0 + 32 * q + lane] : 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) sf = fmaf(x[q], x[q], sf);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sf += __shfl_xor_sync(0xffffffffu, sf, o);
    double s = (double)sf;
    if (!(sf > 1e-30f && sf < 1e30f)) {
        s = 0.0;
        for (int c = lane; c < n; c += 32) s = fma(row[c], row[c], s);
        s = warp_sum_d(s);
    }
    if (lane == 0) {
        const double inv = s > 0x1p-800 ? rsqrt(s) : 0.0, diag = fabs(row[i]);
        rows[i] = {inv, diag, (float)inv, (float)diag};
    }
}

// Whether the pair (i, j) is known well enough, beyond the terms k = i and k = j
// of the sum; false also when another pair has set the flag meanwhile.
__device__ __noinline__ bool small_entry_passes(const double* __restrict__ D, const double* __restrict__ F, int n, int i,
                                                int j, const RowScale& ri, const RowScale& rj, double floor,
                                                const int* flags) {
    const double* di = D + (size_t)i * n;
    const double* dj = D + (size_t)j * n;
    const double d = fabs(di[j]), w = ri.inv * rj.inv;
    if (w == 0.0) return true;
    if (d == 0.0) return F[(size_t)i * n + j] == 0.0;
    double s = d * (ri.diag + rj.diag);
    int k = i;
    for (int c = 0; c < n && s * w < floor; c += 4) {
        if ((c & 63) == 60 && *(const volatile int*)flags) return false;
        double t[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {  // (the loads together)
            const int kk = k + u < n ? k + u : k + u - n;
            t[u] = c + u < n && kk != i && kk != j ? fabs(di[kk] * dj[kk]) : 0.0;
        }
        s += (t[0] + t[1]) + (t[2] + t[3]);
        k = k + 4 < n ? k + 4 : k + 4 - n;
    }
    return s * w >= floor;
}

// Pairs i < j, 32 x 32 at a time, lane: j.  Nearly all pass by their terms k = i and
// k = j; the others add terms from k = i on until they pass.  d_ij = 0 is right
// where F has a zero as well: i and j are then coupled, if at all, through rows
// whose own pairs are tested.  Sets flags[0] at the first pair that does not pass.
__global__ void __launch_bounds__(256)
f64_small_entries_kernel(const double* __restrict__ D, const double* __restrict__ F, int n,
                         const RowScale* __restrict__ rows, int blocks, int step, int* flags) {
    grid_dependency_wait();
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const double floor = 1.0 / (16.0 * n);
    const float quick = (float)floor * 1.0001f;
    for (int b = blockIdx.x; b < blocks; b += gridDim.x) {
        if (*(volatile int*)flags) return;
        int J = (int)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
        while ((J + 1) * (J + 2) / 2 <= b) ++J;
        while (J * (J + 1) / 2 > b) --J;
        const int I = b - J * (J + 1) / 2, j = J * 32 + tx;
        if (j >= n) continue;
        const float inv_j = rows[j].invf, diag_j = rows[j].diagf;
        float d[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = I * 32 + ty + 8 * q;
            d[q] = i < j ? fabsf((float)D[(size_t)i * n + j]) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = I * 32 + ty + 8 * q;
            if (i >= j) continue;
            const float s = d[q] * rows[i].invf * ((rows[i].diagf + diag_j) * inv_j);
            if (s >= quick && s < 1e30f) continue;
            if (!small_entry_passes(D, F, n, i, j, rows[i], rows[j], floor, flags)) atomicCAS(flags, 0, step + 1);
        }
    }
}

size_t plane_bytes(int n_pad) { return (size_t)n_pad * n_pad * kDigits * sizeof(__nv_bfloat16); }
size_t t_bytes(int n_pad) {
    return (size_t)upper_tiles(n_pad / TILE) * TILE * TILE * sizeof(unsigned long long);
}

int ensure_planes(F64Digits& f, int b) {
    if (f.planes[b]) return PURIFY_OK;
    PURIFY_CUDA_TRY(cudaMalloc(&f.planes[b], plane_bytes(f.cap_pad)));
    PURIFY_CUDA_TRY(cudaMalloc(&f.exps[b], sizeof(int) * f.cap_pad));
    return PURIFY_OK;
}

}  // namespace

bool f64d_wanted(int64_t n) { return n >= kF64DigitsMinN && n <= kF64DigitsMaxN; }

double f64d_flops(int64_t n) {
    const double T = pad128(n) / TILE;
    return 43.0 * (T * (T + 1) / 2) * (2.0 * TILE * TILE) * (T * TILE);  // 43 digit pairs
}

bool f64d_begin(F64Digits& f, int64_t n, int operands, long long wait_cycles, cudaStream_t s, int* err) {
    *err = PURIFY_OK;
    if (!f64d_wanted(n)) return false;
    const int n_pad = pad128(n);
    auto ready = [&]() -> int {
        if (n_pad > f.cap_pad) {
            f64d_free(f);
            int dev = 0;
            PURIFY_CUDA_TRY(cudaGetDevice(&dev));
            PURIFY_CUDA_TRY(cudaDeviceGetAttribute(&f.ctas, cudaDevAttrMultiProcessorCount, dev));
            f.cap_pad = n_pad;
            PURIFY_CUDA_TRY(cudaMalloc(&f.T, t_bytes(n_pad)));
            PURIFY_CUDA_TRY(cudaMalloc(&f.flags, 2 * sizeof(int)));
            PURIFY_CUDA_TRY(cudaHostAlloc((void**)&f.host_flags, 2 * sizeof(int), cudaHostAllocDefault));
            PURIFY_CUDA_TRY(cudaMalloc(&f.rows, sizeof(RowScale) * n_pad));
        }
        f.n_pad = n_pad;
        for (int b = 0; b < operands; ++b) PURIFY_TRY(ensure_planes(f, b));
        PURIFY_CUDA_TRY(cudaFuncSetAttribute((const void*)f64_digit_product_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
        if (!f.clean) PURIFY_CUDA_TRY(cudaMemsetAsync(f.T, 0, t_bytes(f.cap_pad), s));
        f.clean = false;
        PURIFY_CUDA_TRY(cudaMemsetAsync(f.flags, 0, 2 * sizeof(int), s));
        return PURIFY_OK;
    };
    const int r = ready();
    f.held[0] = f.held[1] = nullptr;
    f.step = 0;
    f.wait_cycles = wait_cycles > 0 ? wait_cycles : WAIT_CYCLES;
    if (r == PURIFY_OK) return true;
    f64d_free(f);
    if (r == PURIFY_ERR_OOM)
        cudaGetLastError();  // taken: the caller goes on without these buffers
    else
        *err = r;
    return false;
}

static int split_into(F64Digits& f, int b, const double* X, int64_t n, cudaStream_t s) {
    auto go = [&](auto kernel, int rows_per_block) {
        return launch_chained(kernel, (unsigned)(f.n_pad / rows_per_block), 256u, 0, s, X, (int)n, f.n_pad, f.planes[b],
                              f.exps[b], f.flags, f.step);
    };
    PURIFY_CUDA_TRY(n <= 512    ? go(f64_split_kernel<32, 4>, 8)
                    : n <= 1024 ? go(f64_split_kernel<256, 1>, 1)
                    : n <= 4096 ? go(f64_split_kernel<256, 4>, 1)
                                : go(f64_split_kernel<256, 0>, 1));
    count_launches(1);
    f.held[b] = X;
    return PURIFY_OK;
}

int f64d_step(F64Digits& f, const double* A, const double* B, const double* E, double* C, int64_t n, double cP,
              double cE, double cI, double dY, double dI, double* red, cudaStream_t s) {
    f.clean = f.read = false;  // until a check has found every step so far complete
    auto place = [&](const double* X, const double* other, int* b) -> int {
        for (int q = 0; q < 2; ++q)
            if (f.held[q] == X) {
                *b = q;
                return PURIFY_OK;
            }
        *b = (f.held[0] == other && other) ? 1 : 0;
        return split_into(f, *b, X, n, s);
    };
    int a = 0, b = 0;
    PURIFY_TRY(place(A, B, &a));
    if (B == A)
        b = a;
    else
        PURIFY_TRY(place(B, A, &b));
    F64Product L;
    PURIFY_TRY(make_quad_map(&L.map_a, f.planes[a], f.n_pad));
    PURIFY_TRY(make_quad_map(&L.map_b, f.planes[b], f.n_pad));
    L.T = f.T;
    L.flags = f.flags;
    L.wait_cycles = f.wait_cycles;
    L.tiles_per_row = f.n_pad / TILE;
    L.tiles = (int)upper_tiles(L.tiles_per_row);
    int grid = f.ctas;
    L.whole = L.tiles / grid;
    if (L.whole == 0) {
        const long long cost = (long long)L.tiles * L.tiles_per_row * 4 * kCost32;
        grid = (int)std::max<long long>(1, std::min<long long>(grid, cost / kMinCost));
    }
    PURIFY_CUDA_TRY(launch_chained(f64_digit_product_kernel, (unsigned)grid, (unsigned)kThreads, kSmemBytes, s, L));
    const int64_t nb = (n + 31) / 32, blocks = nb * (nb + 1) / 2;
    auto finish = [&](auto kernel, int64_t pieces) {
        return launch_chained(kernel, (unsigned)std::min<int64_t>(pieces, (int64_t)f.ctas * 4), 256u, 0, s, (uint2*)f.T,
                              f.exps[a], f.exps[b], E, C, (int)n, (int)pieces, cP, cE, cI, dY, dI, red, f.flags);
    };
    auto finish_nq = [&](auto e, auto affine) {
        constexpr bool HE = decltype(e)::value, AF = decltype(affine)::value;
        return blocks < 4 * f.ctas ? finish(f64_finish_kernel<1, HE, AF>, 4 * blocks)
                                   : finish(f64_finish_kernel<4, HE, AF>, blocks);
    };
    const bool affine = dY != 1.0 || dI != 0.0;
    PURIFY_CUDA_TRY(E ? (affine ? finish_nq(std::true_type(), std::true_type())
                                : finish_nq(std::true_type(), std::false_type()))
                      : (affine ? finish_nq(std::false_type(), std::true_type())
                                : finish_nq(std::false_type(), std::false_type())));
    count_launches(2);
    for (int q = 0; q < 2; ++q)
        if (f.held[q] == C) f.held[q] = nullptr;
    ++f.step;
    return PURIFY_OK;
}

int f64d_test_entries(F64Digits& f, const double* D, const double* F, int64_t n, cudaStream_t s) {
    if (f.step == 0) return PURIFY_OK;  // no product
    const int64_t nb = (n + 31) / 32, blocks = nb * (nb + 1) / 2;
    PURIFY_CUDA_TRY(launch_chained(f64_row_scale_kernel, (unsigned)((n + 7) / 8), 256u, 0, s, D, (int)n, (RowScale*)f.rows,
                                   f.flags));
    PURIFY_CUDA_TRY(launch_chained(f64_small_entries_kernel, (unsigned)std::min<int64_t>(blocks, (int64_t)f.ctas * 8), 256u, 0,
                                   s, D, F, (int)n, (const RowScale*)f.rows, (int)blocks, f.step, f.flags));
    count_launches(2);
    return PURIFY_OK;
}

int f64d_read(F64Digits& f, cudaStream_t s) {
    PURIFY_CUDA_TRY(cudaMemcpyAsync(f.host_flags, f.flags, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
    f.read = true;
    return PURIFY_OK;
}

int f64d_check(F64Digits& f, int* redo_from, int* wait_flag) {
    *redo_from = -1;
    *wait_flag = 0;
    f.clean = false;
    if (!f.read) return PURIFY_ERR_INTERNAL;
    *wait_flag = f.host_flags[1];
    if (*wait_flag) return PURIFY_ERR_DEVICE_TIMEOUT;
    *redo_from = f.host_flags[0] - 1;
    f.clean = f.host_flags[0] == 0;
    return PURIFY_OK;
}

// 1 GiB holds one operand up to n = 7296, two up to 5376. The allocation is 1 % of a
// run beyond that (n = 8192: 1.3 GiB, 1.6 of 183 ms).
constexpr size_t kF64KeepBytes = 1ull << 30;

void f64d_end(F64Digits& f) {
    if (!f.cap_pad) return;
    const size_t planes = (f.planes[0] ? 1 : 0) + (f.planes[1] ? 1 : 0);
    if (planes * plane_bytes(f.cap_pad) + t_bytes(f.cap_pad) > kF64KeepBytes) f64d_free(f);
}

void f64d_free(F64Digits& f) {
    for (int b = 0; b < 2; ++b) {
        cudaFree(f.planes[b]);
        cudaFree(f.exps[b]);
    }
    cudaFree(f.T);
    cudaFree(f.flags);
    if (f.host_flags) cudaFreeHost(f.host_flags);
    cudaFree(f.rows);
    f = F64Digits();
}

}  // namespace purify
