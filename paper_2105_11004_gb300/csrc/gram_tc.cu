// G = A^T A (d x d, FP64 grade) of a tall FP32 matrix on the tensor cores (tcgen05, sm_103a), by an
// error-free splitting of the entries into BF16 digits.
//
// FP64 runs at 1/64 of the FP32 rate here and the compensated FP32 dot product (k_gram_dot2 in
// gramqr.cu) is bound by FP32 issue at about ten instructions a product. BF16 products are exact and
// an FP32 accumulator holds every integer up to 2^24, so a product of digit matrices is exact as long
// as its chain is short enough:
//   * over a unit's rows, column c is scaled by a power of two, y = x 2^(7 - e_c) with |x| < 2^(e_c), and cut
//     into seven signed digits of 8 bits, y = sum_i t_i with t_i a multiple of 2^(-8i) and |t_i| <= 2^(7 - 8i)
//     (i > 0: at most half a unit of digit i - 1). Each t_i is a BF16 number; what is left after the seventh
//     digit is below 2^-56 of the column's largest entry (a 24-bit entry leaves nothing unless it is
//     smaller than 2^-32 of it);
//   * the products t_i t_j with i + j = g are multiples of 2^(-8g) of at most 2^(14 - 8g). A 24-bit entry has
//     at most four digits that are not zero, in a row (its first at i0: it is at least 2^(-8 i0 - 1), a multiple
//     of 2^(-8 i0 - 24), so digit i0 + 3 leaves nothing), so a row has at most four of these products, and over
//     a chunk of 256 rows the sum stays inside 24 bits: the accumulators of g = 0 .. 6 are exact. Pairs with
//     i + j > 6 are dropped (2^-56);
//   * every 256 rows the accumulators join a running FP32 pair per entry of the tile. The pair drifts with the
//     length of its sum (each of a chunk's seven additions rounds at 2^-48 of it, the same way where rows repeat:
//     constant columns were 4.8e-13 off after 341 chunks, 1.4e-11 after 9,766), so it joins an FP64 number every
//     8 chunks; the partial sums of the row splits are scaled back (powers of two) and added in FP64 in a fixed
//     order.
// Largest error of an entry against a 64-bit product, relative to sqrt(G_ii G_jj) (the compensated sums' in
// brackets): 7.0e-15 at 4096 x 1024 Gaussian (1.1e-14), 2.0e-14 with rows scaled by e^(2 N) (9.7e-14); 1.7e-15 at
// 1e6 x 256 Gaussian (5.1e-15), 4.5e-15 with rank 200 and e^(2 N) (1.1e-14), 1.5e-14 with e^(4 N) (8.9e-15); 3.3e-15
// at 100,003 x 500 (4.6e-15), 3.2e-15 at 80,000 x 1,024 with a quarter of the entries (4.7e-15), 4.0e-14 at
// 1e6 x 1,024 with constant columns (8.9e-13).
//
// Equal columns give bitwise equal rows and columns of G, as the symmetric compensated sums do (a pivot tie
// goes to the lower index): the chunk sums are exact, and every tile has the same chunks and row splits, so
// an entry's roundings do not depend on the tile it lies in.
//
// One CTA takes a 128 x 128 tile of G over a range of rows. 512 accumulator columns hold four 128 x 128
// accumulators, and seven are needed: a chunk runs twice through the ring of stages, first for g = 0 .. 3 (four
// digits), then for g = 4 .. 6 (seven digits); converting twice costs less than smaller tiles, whose MMAs
// would wait for shared memory (a 128 x 128 x 16 MMA already reads its 128 bytes a cycle). A tile of the
// diagonal has one operand to convert and takes three quarters of the time of another.
//   * warps 8..15 (converters): thread = column; read 16 rows of the column two half steps ahead (cp.async,
//     any alignment), cut them into digits and store each digit's 16-byte pieces into the stage (K-major rows
//     of 32 bytes, 32-byte swizzle);
//   * warp 16: allocates tensor memory and issues the MMAs (M = N = 128, K = 16);
//   * warps 0..7 (fetchers): TMEM lane = row of the tile, 64 columns a warp; add a pass's accumulators to the
//     running pairs and hand each accumulator back as soon as it is read.
// The converters set the pace (two warps a scheduler; the tensor pipe is active 40% of the time at 4096 x 1024):
// 2.19 ms at 1e6 x 256, with the column maxima 0.15 ms and the sum of the splits 0.02 ms, against 14.9 ms for
// the compensated sums; 0.14 + 0.03 ms at 4096 x 1024 against 0.96 ms. The FP64 additions every 8 chunks cost less
// than the runs differ (2.36 and 2.37 ms in all at 1e6 x 256, 2.63 and 2.64 at 80,000 x 1,024). Every wait is bounded; after a timeout the CTA runs on without waiting (its
// barriers stay matched) and records the failure in the status word.
#include <atomic>
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "f32x2.cuh"
#include "lev_common.cuh"
#include "lev_kernels.cuh"
#include "tc_common.cuh"

namespace lev {
namespace {

using namespace tcx;

constexpr int kTile = 128;
constexpr int kStages = 3;
constexpr int kDigits = 7;
constexpr int kStageBytes = kDigits * 2 * kTile * 32;       // 56 KB: seven digits of 256 columns x 16 rows
constexpr int kFetchWarps = 8, kConvWarps = 8;               // two warpgroups each; the fifth holds the MMA warp
constexpr int kMmaWarp = kFetchWarps + kConvWarps;
constexpr int kThreads = (kMmaWarp + 4) * 32;
constexpr int kConvThreads = kConvWarps * 32;
constexpr int kMaxChunk = 256;
constexpr int kHalf = 8;                                    // rows of its column a worker converts at a time
constexpr int kRing = 3;                                   // half steps of a thread's column, read two ahead
constexpr int kSlotFloats = kHalf * kConvThreads;
constexpr int kRingBytes = kRing * kSlotFloats * 4;
constexpr int kMaxRows = 128;                               // rows of a block of column maxima
constexpr int kFlush = 8;                                   // chunks after which a tile's pairs join FP64 numbers
constexpr int kUnitDoubles = kTile * kTile + kTile;        // a unit's partial tile (FP64, or FP32 pairs) and 256 exponents
constexpr uint64_t kWaitNs = 2000000000ull;
constexpr int32_t kStatusGramTimeout = 5;

struct GramCtl {
    uint64_t full[kStages], empty[kStages], tfull, afree[4];
    uint32_t tmem_base;
    int32_t abort;
    uint32_t colall[2 * kTile];                            // the columns' maxima
};

// Bounded wait; after a timeout (this one or an earlier one) every wait returns at once.
__device__ __forceinline__ void wait_or_abort(uint32_t bar, uint32_t parity, GramCtl* ctl, int32_t* status) {
    if (mbar_try_wait(bar, parity)) return;
    const uint64_t t0 = global_ns();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return;
        if ((it & 63u) == 0) {
            if (*(volatile int32_t*)&ctl->abort) return;
            if (global_ns() - t0 > kWaitNs) {
                *(volatile int32_t*)&ctl->abort = 1;
                atomicExch(status, kStatusGramTimeout);
                return;
            }
        }
    }
}

// K-major operand with rows of 32 bytes (16 BF16), 32-byte swizzle: 8-row groups 256 bytes apart.
__device__ __forceinline__ uint64_t sw32_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1u << 16;
    d |= (uint64_t)(256u >> 4) << 32;
    d |= (uint64_t)1u << 46;
    d |= (uint64_t)6u << 61;                               // SWIZZLE_32B
    return d;
}

// 2^e with |x| < 2^e for the largest |x| of a column (its FP32 bits). Columns below 2^-119 (whose
// squares are zero in FP32) share one scale; a non-finite entry makes its digits, and so its row and
// column of G, NaN.
__device__ __forceinline__ int column_exponent(uint32_t maxbits) {
    const int e = (int)(maxbits >> 23) - 126;
    return e < -119 ? -119 : e;
}
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }

__device__ __forceinline__ void store_digit(uint8_t* dst, const f32x2 (&t)[4]) {
    uint4 v;
    uint32_t* w = reinterpret_cast<uint32_t*>(&v);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float lo, hi;
        unpack2(t[k], lo, hi);
        const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
        w[k] = *reinterpret_cast<const uint32_t*>(&p);
    }
    *reinterpret_cast<uint4*>(dst) = v;
}

// Eight scaled entries into N digits (slice q at dst + q * slice_bytes).
template <int N>
__device__ __forceinline__ void cut_digits(f32x2 (&y)[4], uint8_t* dst, int slice_bytes) {
    float magic = 12582912.0f;                             // 1.5 2^23: y + magic - magic rounds y to an integer
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const f32x2 mg = pack2(magic, magic);
        f32x2 t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            t[k] = sub2(add2(y[k], mg), mg);
            if (q + 1 < N) y[k] = sub2(y[k], t[k]);
        }
        store_digit(dst + q * slice_bytes, t);
        magic *= 0.00390625f;
    }
}

struct GramPlan {
    int nt, noff;              // 128-column blocks, tiles above the diagonal
    int splits, rows;          // row splits of every tile, rows a split
    int chunk;                 // rows a chunk (multiple of 16, at most kMaxChunk)
    int flush;                 // kFlush where a split has more chunks (partial tiles in FP64), else 0 (FP32 pairs)
};

__device__ __forceinline__ void off_tile(int t, int nt, int& bi, int& bj) {
    bi = 0;
    while (t >= nt - 1 - bi) { t -= nt - 1 - bi; ++bi; }
    bj = bi + 1 + t;
}

// The MMAs of one K step for pass 0 (g = 0 .. 3, accumulator g) or pass 1 (g = 4 .. 6, accumulator g - 4). sa: stage address (digit 0 of the tile's rows); the operands of the tile's
// columns follow them, or are the same rows (a tile of the diagonal). `first`: the pass's first step (the
// accumulators start at zero, and each is waited for). One thread issues them, so the operand
// addresses are constants off one descriptor.
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r;
}
// tcgen05.mma by the thread with lead != 0, in code that the whole warp runs: the operands stay in uniform
// registers (inside an `if (lane == 0)` each was moved there anew, 160 cycles an MMA against 64 of work).
__device__ __forceinline__ void mma_if(uint32_t lead, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum), "r"(lead)
        : "memory");
}

template <bool DIAG, int PASS, class WaitAcc>
__device__ __forceinline__ void issue_step(uint32_t lead, uint32_t sa, uint32_t tmem, bool first, WaitAcc wait_acc) {
    constexpr uint32_t kSlice = (DIAG ? 1u : 2u) * kTile * 32u, idesc = make_idesc(false, kTile, kTile);
    const uint64_t a = sw32_desc(sa), b = a + (DIAG ? 0u : kTile * 32u / 16u);
#pragma unroll
    for (int acc = 0; acc < (PASS == 0 ? 4 : 3); ++acc) {
        const int g = 4 * PASS + acc;
        if (first) wait_acc(acc);
#pragma unroll
        for (int i = 0; i <= g; ++i)
            mma_if(lead, tmem + (uint32_t)acc * kTile, a + (uint32_t)i * (kSlice / 16u), b + (uint32_t)(g - i) * (kSlice / 16u),
                   idesc, (i == 0 && first) ? 0u : 1u);
    }
}

// out[q][c] = the largest |A[i][c]| (as FP32 bits) of rows 128 q .. 128 q + 127. A pass of its own: inside
// k_gram_tc too few loads are in flight to stream the rows (1.5 ms at 1e6 x 256 against 0.17).
__global__ void __launch_bounds__(512) k_gram_colmax(const float* __restrict__ A, int64_t lda, int64_t m, int d,
                                                     uint32_t* __restrict__ out) {
    __shared__ uint32_t part[4][kTile];
    const int c = threadIdx.x & (kTile - 1), g = threadIdx.x >> 7;
    const int64_t col = (int64_t)blockIdx.y * kTile + c, r0 = (int64_t)blockIdx.x * kMaxRows;
    const int rows = (int)min((int64_t)kMaxRows, m - r0);
    uint32_t mx = 0;
    if (col < d) {
        const float* src = A + r0 * lda + col;
        int r = g;
        for (; r + 28 < rows; r += 32) {
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = __ldg(src + (r + 4 * e) * lda);
#pragma unroll
            for (int e = 0; e < 8; ++e) mx = max(mx, __float_as_uint(v[e]) & 0x7fffffffu);
        }
        for (; r < rows; r += 4) mx = max(mx, __float_as_uint(__ldg(src + r * lda)) & 0x7fffffffu);
    }
    part[g][c] = mx;
    __syncthreads();
    if (g == 0 && col < d)
        out[blockIdx.x * (int64_t)d + col] = max(max(part[0][c], part[1][c]), max(part[2][c], part[3][c]));
}

// x 2^k as a double, by its bits (FP64 conversions and multiplies run at 1/64 of the integer rate): x zero,
// normal or not finite; -252 <= k <= 244.
__device__ __forceinline__ double scaled_double(float x, int k) {
    const uint32_t b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    const uint32_t hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + ((uint32_t)(896 + k) << 20));
    if (e == 0xffu) return __hiloint2double(0x7ff80000, 0);
    return e == 0 ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}

__global__ void __launch_bounds__(kThreads, 1) k_gram_tc(const float* __restrict__ A, int64_t lda, int64_t m, int d,
                                                         GramPlan pl, const uint32_t* __restrict__ colmax, double* __restrict__ Gp,
                                                         int32_t* status) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* base = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    GramCtl* ctl = reinterpret_cast<GramCtl*>(base + kStages * kStageBytes + kRingBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // unit: a tile and a range of rows; tiles above the diagonal first
    int bi, bj, split;
    const bool diag = (int)blockIdx.x >= pl.noff * pl.splits;
    if (!diag) {
        split = (int)blockIdx.x / pl.noff;
        off_tile((int)blockIdx.x % pl.noff, pl.nt, bi, bj);
    } else {
        const int u = (int)blockIdx.x - pl.noff * pl.splits;
        split = u / pl.nt;
        bi = bj = u % pl.nt;
    }
    const int K = pl.chunk;
    const int64_t r_begin = min(m, (int64_t)split * pl.rows), r_end = min(m, r_begin + pl.rows);
    const int ns = K / 16;                                 // K steps a pass
    const int nchunk = (int)((r_end - r_begin + K - 1) / K);
    const int nseg = 2 * nchunk;                           // passes
    const int slice = (diag ? 1 : 2) * kTile * 32;          // bytes a digit

    if (threadIdx.x == 0) {
        for (int q = 0; q < kStages; ++q) {
            mbar_init(smem_u32(&ctl->full[q]), diag ? 4 : 8);
            mbar_init(smem_u32(&ctl->empty[q]), 1);
        }
        mbar_init(smem_u32(&ctl->tfull), 1);
        for (int q = 0; q < 4; ++q) mbar_init(smem_u32(&ctl->afree[q]), kFetchWarps);
        ctl->abort = 0;
        fence_mbar_init();
    }
    // columns past d are never written: their operand rows stay zero
    for (int e = threadIdx.x; e < kStages * kStageBytes / 16; e += kThreads)
        reinterpret_cast<uint4*>(base)[e] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
    __syncthreads();
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32(&ctl->tmem_base), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    double* unit = Gp + (int64_t)blockIdx.x * kUnitDoubles;

    if (warp >= kMmaWarp) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
        if (warp == kMmaWarp && nseg > 0) {
            const uint32_t lead = elect_one();
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0), base_u = __shfl_sync(0xffffffffu, smem_u32(base), 0);
            int s = 0;
            uint32_t phase = 0;
            for (int seg = 0; seg < nseg; ++seg) {
                auto wait_acc = [&](int a) {
                    if (seg > 0) {
                        wait_or_abort(smem_u32(&ctl->afree[a]), (uint32_t)((seg - 1) & 1), ctl, status);
                        __syncwarp();
                        tc_fence_after();
                    }
                };
                for (int step = 0; step < ns; ++step) {
                    wait_or_abort(smem_u32(&ctl->full[s]), phase, ctl, status);
                    __syncwarp();
                    tc_fence_after();
                    const uint32_t a = base_u + (uint32_t)s * kStageBytes;
                    if (diag) {
                        if (seg & 1) issue_step<true, 1>(lead, a, tm, step == 0, wait_acc);
                        else issue_step<true, 0>(lead, a, tm, step == 0, wait_acc);
                    } else {
                        if (seg & 1) issue_step<false, 1>(lead, a, tm, step == 0, wait_acc);
                        else issue_step<false, 0>(lead, a, tm, step == 0, wait_acc);
                    }
                    if (lead) tc_commit(smem_u32(&ctl->empty[s]));
                    __syncwarp();
                    if (++s == kStages) { s = 0; phase ^= 1u; }
                }
                if (lead) tc_commit(smem_u32(&ctl->tfull));
                __syncwarp();
            }
            // every MMA has finished before tensor memory is freed
            wait_or_abort(smem_u32(&ctl->tfull), (uint32_t)((nseg - 1) & 1), ctl, status);
            __syncwarp();
        }
    } else if (warp >= kFetchWarps) {
        // ---- converters: two groups of 128 threads, thread = column of a block of 128. Group g takes block g of
        // every K step (rows' and columns' operand), or in a tile of the diagonal (one block) every other step
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        const int t = threadIdx.x - kFetchWarps * 32, grp = t >> 7, c = t & (kTile - 1);
        const int nb = diag ? 1 : 2;                        // blocks a step
        const int colb0 = bi * kTile + c, bstep = (bj - bi) * kTile;   // column in the first block, to the second
        // the largest entry of each column over the unit's rows (k_gram_colmax's blocks that hold them): one
        // power of two scales the column
        if (!diag || grp == 0) {
            const int cc = colb0 + grp * bstep;
            uint32_t mx = 0;
            if (cc < d && r_begin < r_end)
                for (int64_t q = r_begin / kMaxRows; q <= (r_end - 1) / kMaxRows; ++q) mx = max(mx, colmax[q * d + cc]);
            ctl->colall[grp * kTile + c] = mx;
            if (diag) ctl->colall[kTile + c] = mx;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kConvThreads) : "memory");
        const int b = diag ? 0 : grp, stride = diag ? 2 : 1, first = diag ? grp : 0;
        const int col = colb0 + b * bstep;
        const bool ok = col < d, live = __any_sync(0xffffffffu, ok);
        const float scale = pow2f(7 - column_exponent(ctl->colall[b * kTile + c]));
        const uint32_t ring = smem_u32(base + kStages * kStageBytes) + 4 * t;
        // the thread's half steps (8 rows of its column) in order, read two ahead into its own part of the ring
        struct Pos { int u, step, pass, row; };             // K step of the unit, step of its pass, first row of its chunk
        auto norm = [&](Pos& p) {
            while (p.step >= ns) {
                p.step -= ns;
                p.row += p.pass ? K : 0;
                p.pass ^= 1;
            }
        };
        Pos at = {first, first, 0, 0};                      // next to convert
        norm(at);
        Pos rd = at;                                       // next to read
        int rhalf = 0;
        const int nrows = (int)(r_end - r_begin), nsteps = nseg * ns;
        const float* acol = A + r_begin * lda + (ok ? col : 0);
        auto read_half = [&](int slot) {
            const int row = rd.row + rd.step * 16 + rhalf * kHalf;
            const int left = rd.u < nsteps && ok ? nrows - row : 0;
            uint32_t to = ring + (uint32_t)slot * (kSlotFloats * 4);
            const float* p = acol + (left > 0 ? row * lda : 0);
            if (left >= kHalf) {
#pragma unroll
                for (int k = 0; k < kHalf; ++k) {
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to + k * (kConvThreads * 4)), "l"(p) : "memory");
                    p += lda;
                }
            } else {
#pragma unroll 1
                for (int k = 0; k < kHalf; ++k) {
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(to), "l"(k < left ? p : A),
                                 "r"(k < left ? 4 : 0)
                                 : "memory");
                    p += lda;
                    to += kConvThreads * 4;
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            if ((rhalf ^= 1) == 0) {
                rd.u += stride;
                rd.step += stride;
                norm(rd);
            }
        };
#pragma unroll 1
        for (int q = 0; q < kRing - 1; ++q) read_half(q);
        int slot = 0;
        const int swz = ((c >> 2) & 1) << 4;
        while (at.u < nsteps) {
            const int s = at.u % kStages;
            uint8_t* to = base + s * kStageBytes + (b * kTile + c) * 32;
            wait_or_abort(smem_u32(&ctl->empty[s]), (uint32_t)((at.u / kStages) & 1) ^ 1u, ctl, status);
            __syncwarp();
#pragma unroll 1
            for (int hh = 0; hh < 2; ++hh) {
                read_half(slot == 0 ? kRing - 1 : slot - 1);
                asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 1) : "memory");
                if (live) {
                    f32x2 x[kHalf / 2];
                    const f32x2 sc = pack2(scale, scale);
                    const uint32_t from = ring + (uint32_t)slot * (kSlotFloats * 4);
#pragma unroll
                    for (int k = 0; k < kHalf / 2; ++k) {
                        float a0, a1;
                        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(a0) : "r"(from + 2 * k * (kConvThreads * 4)) : "memory");
                        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(a1) : "r"(from + (2 * k + 1) * (kConvThreads * 4)) : "memory");
                        x[k] = mul2(pack2(a0, a1), sc);
                    }
                    if (at.pass == 0) cut_digits<4>(x, to + ((hh << 4) ^ swz), slice);
                    else cut_digits<kDigits>(x, to + ((hh << 4) ^ swz), slice);
                }
                if (++slot == kRing) slot = 0;
            }
            if (live) fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl->full[s]));
            at.u += stride;
            at.step += stride;
            norm(at);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else {
        // ---- fetchers: warp w holds rows 32 (w mod 4) + lane, columns 64 (w / 4) .. + 63 of the tile as FP32
        // pairs (256 x 168 + 256 x 56 + 128 x 32 = 640 x 96 registers, the block's at launch)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
        const int lq = warp & 3, cg = warp >> 2;
        const uint32_t tacc = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(cg * 64);
        double* out = unit + (cg * 64) * kTile + lq * 32 + lane;   // column-major (lanes write consecutive rows)
        if (pl.flush)
            for (int j = 0; j < 64; ++j) out[j * kTile] = 0.0;
        int seg = 0;
        do {                                               // the chunks of one running pair
            f32x2 h[32], l[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) h[j] = l[j] = 0ull;
            const int end = pl.flush ? min(nseg, seg + 2 * kFlush) : nseg;
            for (; seg < end; ++seg) {
                // add the pass's accumulators: error-free for g <= 3; the sums of g >= 4 (about 2^-27 of the largest
                // entry's square) join the low parts
                const int pass = seg & 1;
                wait_or_abort(smem_u32(&ctl->tfull), (uint32_t)(seg & 1), ctl, status);
                __syncwarp();
                tc_fence_after();
                const int nacc = pass == 0 ? 4 : 3;
                for (int a = 0; a < nacc; ++a) {
#pragma unroll
                    for (int j0 = 0; j0 < 64; j0 += 8) {
                        uint32_t r[8];
                        tmem_ld8(tacc + (uint32_t)(a * kTile + j0), r);
                        tmem_ld_wait();
                        if (j0 == 56) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) {
                                mbar_arrive(smem_u32(&ctl->afree[a]));
                                if (pass == 1 && a == 2) mbar_arrive(smem_u32(&ctl->afree[3]));
                            }
                        }
                        if (pass == 0) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                f32x2& hj = h[j0 / 2 + j];
                                const f32x2 v = pack2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
                                const f32x2 s1 = add2(hj, v), z = sub2(s1, hj);
                                const f32x2 er = add2(sub2(hj, sub2(s1, z)), sub2(v, z));   // h + v = s1 + er
                                hj = s1;
                                l[j0 / 2 + j] = add2(l[j0 / 2 + j], er);
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                l[j0 / 2 + j] = add2(l[j0 / 2 + j], pack2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1])));
                        }
                    }
                }
                if (pass == 1) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const f32x2 s1 = add2(h[j], l[j]), z = sub2(s1, h[j]);
                        l[j] = add2(sub2(h[j], sub2(s1, z)), sub2(l[j], z));
                        h[j] = s1;
                    }
                }
            }
            // the pairs as they are, or into the partial tile's FP64 numbers (this thread's alone: the additions
            // in L2 come in its order, and nothing waits for them)
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                float h0, h1, l0, l1;
                unpack2(h[j], h0, h1);
                unpack2(l[j], l0, l1);
                if (pl.flush) {
                    atomicAdd(out + 2 * j * kTile, scaled_double(h0, 0) + scaled_double(l0, 0));
                    atomicAdd(out + (2 * j + 1) * kTile, scaled_double(h1, 0) + scaled_double(l1, 0));
                } else {
                    reinterpret_cast<float2*>(out)[2 * j * kTile] = make_float2(h0, l0);
                    reinterpret_cast<float2*>(out)[(2 * j + 1) * kTile] = make_float2(h1, l1);
                }
            }
        } while (seg < nseg);
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 2 * kTile)                           // the columns' exponents, rows' block first
        reinterpret_cast<int32_t*>(unit + kTile * kTile)[threadIdx.x] = column_exponent(ctl->colall[threadIdx.x]);
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// G (d x d, both triangles) from the units' partials: scaled back and added in FP64. A CTA takes a 32 x 4
// block of a tile (blockIdx.y: block row + 4 block column); warp w adds the splits w, w + 8, ... of its four
// columns, then the warps' sums are added in warp order.
__global__ void __launch_bounds__(256) k_gram_tc_reduce(const double* __restrict__ Gp, int d, GramPlan pl,
                                                        double* __restrict__ G) {
    constexpr int T = kTile * kTile;
    __shared__ double part[8][4][33];
    const int tile = blockIdx.x, r0 = (blockIdx.y & 3) * 32, c0 = (blockIdx.y >> 2) * 4;
    const bool diag = tile >= pl.noff;
    if (diag && r0 > c0 + 3) return;
    int bi, bj;
    if (diag) bi = bj = tile - pl.noff;
    else off_tile(tile, pl.nt, bi, bj);
    const double* p = Gp + (int64_t)(diag ? pl.noff * pl.splits + bi : tile) * kUnitDoubles;
    const int64_t stride = (int64_t)(diag ? pl.nt : pl.noff) * kUnitDoubles;
    const int tx = threadIdx.x & 31, w = threadIdx.x >> 5;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
    for (int z = w; z < pl.splits; z += 8) {
        const double* u = p + z * stride;
        const int32_t* ex = reinterpret_cast<const int32_t*>(u + T);
        const int er = ex[r0 + tx] - 14;
        double x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = u[(c0 + q) * kTile + r0 + tx];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k = er + ex[kTile + c0 + q];
            if (pl.flush) {
                s[q] += x[q] * __hiloint2double((1023 + k) << 20, 0);
            } else {                                        // the pair (high part in the low word)
                s[q] += scaled_double(__int_as_float(__double2loint(x[q])), k);
                s[q] += scaled_double(__int_as_float(__double2hiint(x[q])), k);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) part[w][q][tx] = s[q];
    __syncthreads();
    // warp w < 4: column w of the block
    const int gi = bi * kTile + r0 + tx, gj = bj * kTile + c0 + w;
    if (w < 4 && gi < d && gj < d && !(diag && gi > gj)) {
        double t = 0.0;
#pragma unroll
        for (int v = 0; v < 8; ++v) t += part[v][w][tx];
        G[(int64_t)gj * d + gi] = t;
        G[(int64_t)gi * d + gj] = t;
    }
}

int device_sms() {
    static std::atomic<int> cached{0};                     // host threads share it
    int sms = cached.load(std::memory_order_relaxed);
    if (sms == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
            sms = 152;
        cached.store(sms, std::memory_order_relaxed);
    }
    return sms;
}

// Row splits, the same for every tile: the count with the shortest schedule of at most three CTAs an SM, at
// least 64 rows a split. In quarters of the time of a tile above the diagonal (0.124 us a row), one on the
// diagonal takes three (0.094 us: its converters have half the work, the MMAs and fetches are the same), and
// starting and ending a CTA about 260 rows. CTAs start in the order of their index, the long ones first. At
// 1e6 x 256 that is 152 splits, every SM with one tile above and two on the diagonal (2.05 ms when the counts were
// compared; 2.46 with 76 splits, 2.39 with 50 in one wave).
GramPlan make_plan(int64_t m, int64_t d) {
    const int64_t sms = device_sms();
    GramPlan p;
    p.nt = (int)((d + kTile - 1) / kTile);
    p.noff = p.nt * (p.nt - 1) / 2;
    const int64_t most = std::max<int64_t>(1, std::min((m + 63) / 64, 3 * sms / (p.noff + p.nt)));
    auto rows = [&](int64_t s) { return ((m + s - 1) / s + 15) / 16 * 16; };
    int64_t best = INT64_MAX;
    p.splits = 1;
    for (int64_t s = 1; s <= most; ++s) {
        const int64_t off = p.noff * s, dia = p.nt * s;
        // the SMs end the long units at `t0` (`late` of them at t0 + 4); time for the others after that
        const int64_t t0 = off / sms * 4, late = off % sms;
        int64_t t = late ? 4 : 0;
        while (late * ((t >= 4 ? t - 4 : 0) / 3) + (sms - late) * (t / 3) < dia) ++t;
        const int64_t cost = (t0 + t) * rows(s) + 260 * ((off + dia + sms - 1) / sms);
        if (cost < best) {
            best = cost;
            p.splits = (int)s;
        }
    }
    p.rows = (int)rows(p.splits);
    p.splits = (int)std::max<int64_t>(1, (m + p.rows - 1) / p.rows);
    const int n = (p.rows + kMaxChunk - 1) / kMaxChunk;
    p.chunk = std::min(kMaxChunk, ((p.rows + n - 1) / n + 15) / 16 * 16);
    p.flush = (p.rows + p.chunk - 1) / p.chunk > kFlush ? kFlush : 0;
    return p;
}

size_t colmax_doubles(int64_t m, int64_t d) { return (size_t)(((m + kMaxRows - 1) / kMaxRows * d + 1) / 2); }

}  // namespace

size_t gram_tc_partial_doubles(int64_t m, int64_t d) {
    const GramPlan p = make_plan(m, d);
    return (size_t)(p.noff + p.nt) * p.splits * kUnitDoubles + colmax_doubles(m, d);
}

cudaError_t launch_gram_tc(const float* A, int64_t lda, int64_t m, int64_t d, double* Gp, double* G, int32_t* status,
                           cudaStream_t st) {
    const GramPlan p = make_plan(m, d);
    const size_t smem = 1024 + (size_t)kStages * kStageBytes + kRingBytes + sizeof(GramCtl);
    cudaError_t e = cudaFuncSetAttribute(k_gram_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const unsigned units = (unsigned)((p.noff + p.nt) * p.splits);
    uint32_t* colmax = reinterpret_cast<uint32_t*>(Gp + (size_t)units * kUnitDoubles);
    k_gram_colmax<<<dim3((unsigned)((m + kMaxRows - 1) / kMaxRows), (unsigned)p.nt), 512, 0, st>>>(A, lda, m, (int)d, colmax);
    k_gram_tc<<<units, kThreads, smem, st>>>(A, lda, m, (int)d, p, colmax, Gp, status);
    k_gram_tc_reduce<<<dim3((unsigned)(p.noff + p.nt), 128), 256, 0, st>>>(Gp, (int)d, p, G);
    return cudaGetLastError();
}

}  // namespace lev
