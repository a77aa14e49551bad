// Fused final pass theta~_i = ||A_i Mfull||^2 (Alg. 8 step 5), FP32 SIMT forms.
//
// Mfull (d x k) holds R_11^{-1} Omega on the rows of the selected columns K and
// zeros elsewhere, so A Mfull = A_K R_11^{-1} Omega. The n x k product never
// leaves registers: each CTA squares and sums its tile rows in the epilogue
// (warp shuffles) and writes only theta~ (n floats).
//
// Dense: 128-row (64 for small n) x 256-column register tile, 16 x 8 per
// thread, A and Mfull staged through shared memory in 16-wide k slices (two
// stages), packed FP32 FMAs on row pairs.
// CSR, long rows: one warp per row (product form of Lemma 1): the warp broadcasts
// each (col, val) of the row and every lane accumulates 8 columns of
// val * Mfull[col, :] with 128-bit loads; then squares and warp-sums. Short rows:
// the pairs of the row's entries against P = Mfull Mfull^T.
#include "f32x2.cuh"
#include "lev_common.cuh"
#include "lev_kernels.cuh"

namespace lev {

namespace {

constexpr int FD_BN = 256, FD_BK = 16;

// A warp owns 2 NP rows (NP packed pairs), lane l columns 4 l .. + 3 and 128 + 4 l .. + 3. Bound by the FP32
// FMA pipe: with 8 rows a thread (NP = 4) the columns' shared-memory reads, eight wavefronts for 64 FMAs a
// lane, kept the pipe at 0.44 (2.88 ms at 1e6 x 256 x 256); 16 rows halve them. Row pairs are
// packed because the rows' entries are read as pairs anyway (one broadcast a pair); the columns' entries are
// doubled in registers. NP = 4 keeps small n on more SMs. Each sum runs over k in order, as scalar FMAs would.
template <bool VEC, int NP>
__global__ void __launch_bounds__(256, NP == 8 ? 1 : 2) k_final_dense_fp32(
        const float* __restrict__ A, int64_t lda, int64_t n, int d,
        const float* __restrict__ M, int k, float* __restrict__ theta) {
    constexpr int BM = 16 * NP, LD = BM + 4;               // rows of the tile; + 4: the transposed stores' banks
    __shared__ __align__(16) float As[2][FD_BK][LD];
    __shared__ __align__(16) float Ms[2][FD_BK][FD_BN];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int64_t row0 = (int64_t)blockIdx.x * BM;
    // loader coordinates: A tile BM x 16 (NP / 4 float4 per thread), M tile 16 x 256 (4 float4)
    const int a_r = t >> 2, a_c = (t & 3) * 4;
    const int m_r = t >> 4, m_c = (t & 15) * 4;
    float th[2 * NP];
#pragma unroll
    for (int i = 0; i < 2 * NP; ++i) th[i] = 0.f;

    for (int q0 = 0; q0 < k; q0 += FD_BN) {
        f32x2 acc[NP][8];
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
        float ra[NP / 4][4], rm[4][4];
        auto load = [&](int k0) {
#pragma unroll
            for (int u = 0; u < NP / 4; ++u) {
                const int64_t gr = row0 + a_r + 64 * u;
                if (VEC) {
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (gr < n && k0 + a_c < d) v = __ldg(reinterpret_cast<const float4*>(A + gr * lda + k0 + a_c));
                    ra[u][0] = v.x; ra[u][1] = v.y; ra[u][2] = v.z; ra[u][3] = v.w;
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int c = k0 + a_c + i;
                        ra[u][i] = (gr < n && c < d) ? __ldg(A + gr * lda + c) : 0.f;
                    }
                }
            }
            const int mr = k0 + m_r;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = q0 + m_c + 64 * u;
                if (VEC) {
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (mr < d && c < k) v = __ldg(reinterpret_cast<const float4*>(M + (int64_t)mr * k + c));
                    rm[u][0] = v.x; rm[u][1] = v.y; rm[u][2] = v.z; rm[u][3] = v.w;
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        rm[u][i] = (mr < d && c + i < k) ? __ldg(M + (int64_t)mr * k + c + i) : 0.f;
                }
            }
        };
        auto store = [&](int st) {
#pragma unroll
            for (int u = 0; u < NP / 4; ++u)
#pragma unroll
                for (int i = 0; i < 4; ++i) As[st][a_c + i][a_r + 64 * u] = ra[u][i];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                *reinterpret_cast<float4*>(&Ms[st][m_r][m_c + 64 * u]) =
                    make_float4(rm[u][0], rm[u][1], rm[u][2], rm[u][3]);
        };
        int st = 0;
        load(0);
        __syncthreads();                 // previous chunk's readers are done
        store(0);
        __syncthreads();
        for (int k0 = 0; k0 < d; k0 += FD_BK) {
            const bool more = (k0 + FD_BK) < d;
            if (more) load(k0 + FD_BK);
#pragma unroll
            for (int kk = 0; kk < FD_BK; ++kk) {
                f32x2 a[NP];
#pragma unroll
                for (int i = 0; i < NP; i += 2) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&As[st][kk][w * 2 * NP + 2 * i]);
                    a[i] = v.x;
                    a[i + 1] = v.y;
                }
                const float4 b0 = *reinterpret_cast<const float4*>(&Ms[st][kk][lane * 4]);
                const float4 b1 = *reinterpret_cast<const float4*>(&Ms[st][kk][128 + lane * 4]);
                const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const f32x2 bb = pack2(b[j], b[j]);
#pragma unroll
                    for (int i = 0; i < NP; ++i) acc[i][j] = fma2(a[i], bb, acc[i][j]);
                }
            }
            if (more) {
                store(st ^ 1);
                __syncthreads();
                st ^= 1;
            }
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            f32x2 sq = 0ull;
#pragma unroll
            for (int j = 0; j < 8; ++j) sq = fma2(acc[i][j], acc[i][j], sq);
            float s0, s1;
            unpack2(sq, s0, s1);
            th[2 * i] += s0;
            th[2 * i + 1] += s1;
        }
    }
#pragma unroll
    for (int i = 0; i < 2 * NP; ++i) {
        const float v = warp_sum(th[i]);
        const int64_t r = row0 + w * 2 * NP + i;
        if (lane == 0 && r < n) theta[r] = v;
    }
}

// ||a_i M||^2 of one CSR row (entries p0 .. p1), this lane's share (the caller sums the warp): lane
// owns columns q0 + lane*4 + {0..3} and q0 + 128 + lane*4 + {0..3} of each 256-column chunk.
template <bool VEC>
__device__ __forceinline__ float csr_row_norm(int64_t p0, int64_t p1, const int32_t* __restrict__ col,
                                              const float* __restrict__ val, int d, const float* __restrict__ M,
                                              int k, int lane) {
    float total = 0.f;
    for (int q0 = 0; q0 < k; q0 += 256) {
        float y[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) y[j] = 0.f;
        for (int64_t pb = p0; pb < p1; pb += 32) {
            const int cnt = (int)min((int64_t)32, p1 - pb);
            int my_c = -1;
            float my_v = 0.f;
            if (lane < cnt) {
                my_c = col[pb + lane];
                my_v = val[pb + lane];
                if ((unsigned)my_c >= (unsigned)d) { my_c = 0; my_v = 0.f; }
            }
            int u = 0;
            for (; u + 4 <= cnt; u += 4) {
                float4 m0[4], m1[4];
                float vv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int c = __shfl_sync(0xffffffffu, my_c, u + e);
                    vv[e] = __shfl_sync(0xffffffffu, my_v, u + e);
                    const float* Mr = M + (int64_t)c * k + q0;
                    if (VEC) {
                        m0[e] = (q0 + lane * 4 < k) ? __ldg(reinterpret_cast<const float4*>(Mr + lane * 4))
                                                    : make_float4(0.f, 0.f, 0.f, 0.f);
                        m1[e] = (q0 + 128 + lane * 4 < k)
                                    ? __ldg(reinterpret_cast<const float4*>(Mr + 128 + lane * 4))
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
                    } else {
                        float tmp[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int q = q0 + (j < 4 ? lane * 4 + j : 128 + lane * 4 + j - 4);
                            tmp[j] = (q < k) ? __ldg(M + (int64_t)c * k + q) : 0.f;
                        }
                        m0[e] = make_float4(tmp[0], tmp[1], tmp[2], tmp[3]);
                        m1[e] = make_float4(tmp[4], tmp[5], tmp[6], tmp[7]);
                    }
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    y[0] = fmaf(vv[e], m0[e].x, y[0]); y[1] = fmaf(vv[e], m0[e].y, y[1]);
                    y[2] = fmaf(vv[e], m0[e].z, y[2]); y[3] = fmaf(vv[e], m0[e].w, y[3]);
                    y[4] = fmaf(vv[e], m1[e].x, y[4]); y[5] = fmaf(vv[e], m1[e].y, y[5]);
                    y[6] = fmaf(vv[e], m1[e].z, y[6]); y[7] = fmaf(vv[e], m1[e].w, y[7]);
                }
            }
            for (; u < cnt; ++u) {
                const int c = __shfl_sync(0xffffffffu, my_c, u);
                const float v = __shfl_sync(0xffffffffu, my_v, u);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int q = q0 + (j < 4 ? lane * 4 + j : 128 + lane * 4 + j - 4);
                    if (q < k) y[j] = fmaf(v, __ldg(M + (int64_t)c * k + q), y[j]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) total = fmaf(y[j], y[j], total);
    }
    return total;
}

// CSR, warp per row: ||a_i Mfull||^2.
template <bool VEC>
__global__ void __launch_bounds__(256) k_final_csr_fp32(
        const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
        const float* __restrict__ val, int64_t n, int d, const float* __restrict__ M, int k,
        float* __restrict__ theta) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = warp; i < n; i += nwarps) {
        const float total = warp_sum(csr_row_norm<VEC>(row_ptr[i], row_ptr[i + 1], col, val, d, M, k, lane));
        if (lane == 0) theta[i] = total;
    }
}

// CSR with the second form of Lemma 1 for short rows: theta~_i = a_i P a_i^T, P = Mfull Mfull^T
// (d x d), i.e. the sum over the entry pairs p <= q of (2 - [p = q]) a_p a_q P[c_p][c_q]:
// nnz_i^2 / 2 terms from a matrix that sits in L2, against nnz_i k products and nnz_i rows of
// Mfull for the first form. Repeated columns are handled as they stand (the double sum over the
// pairs is the quadratic form); columns outside [0, d) count as zero.
//
// The terms are summed in FP32 arithmetic with double-float accuracy (FP64 runs at 1/64 of the FP32
// rate here and made this pass FP64-bound): P is held as a pair hi + lo of FP32 matrices (the FP64
// Gram matrix of Mfull^T split once), each term's product is formed with its rounding errors
// (TwoProduct of the two entries, the pair of P multiplied in), and every lane accumulates its
// terms with TwoSum, so a row carries an error of a few 2^-48 of sum |terms| rather than 2^-24.
__device__ __forceinline__ void df_add(float& sh, float& sl, float th, float tl) {
    const float s = __fadd_rn(sh, th);
    const float bb = __fsub_rn(s, sh);
    float e = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bb)), __fsub_rn(th, bb));
    e = __fadd_rn(e, __fadd_rn(sl, tl));
    sh = __fadd_rn(s, e);
    sl = __fsub_rn(e, __fsub_rn(sh, s));
}
// (w a b) (P_hi + P_lo) as an unevaluated pair (w = 1 or 2, exact).
__device__ __forceinline__ void df_term(float a, float b, float w, float2 P, float& th, float& tl) {
    const float x = __fmul_rn(a, b);
    const float xe = __fmaf_rn(a, b, -x);                             // a b = x + xe exactly
    const float xw = __fmul_rn(x, w), xwe = __fmul_rn(xe, w);          // exact (w a power of two)
    th = __fmul_rn(xw, P.x);
    tl = __fmaf_rn(xw, P.x, -th);
    tl = __fmaf_rn(xw, P.y, tl);
    tl = __fmaf_rn(xwe, P.x, tl);
}

// Streaming loads of a row's entries: they are read once, so L1 keeps P.
__device__ __forceinline__ int32_t ld_once(const int32_t* p) {
    int32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_once(const float* p) {
    float v;
    asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// The rows of `rows` (bit b: row r0 + b of the warp's 32, each of at most SEG entries; lane b holds its start p0
// and length len), 32 / SEG at a time, SEG lanes a row, the next rows' entries loaded ahead. Lane l of a row
// holds entry l; in step s it takes the pair (l, l + s mod len), so that len / 2 steps visit every pair of two
// entries once with all lanes of the row at work (in the last step of an even length half of them). The
// diagonal terms read dg (P's diagonal, shared memory). Four steps' reads of P are in flight together; their
// terms are formed and summed two at a time with packed instructions, unweighted: the sum over p < q is doubled
// once (exact) before the diagonal terms join it. A product's rounding error is taken against neg2 of the
// rounded product: against a second product with a negated factor the results lost their low parts (2^-25 off).
template <int SEG>
__device__ __forceinline__ void csr_pair_rows(unsigned rows, int64_t p0, int len, int64_t r0, int lane,
                                              const int32_t* __restrict__ col, const float* __restrict__ val, int d,
                                              const float2* __restrict__ P, const float2* dg,
                                              float* __restrict__ theta) {
    if (!rows) return;
    constexpr int RPW = 32 / SEG;
    const int seg = lane / SEG, sl = lane % SEG;
    int b, L, c;
    float a;
    auto fetch = [&]() {
        b = -1;
#pragma unroll
        for (int g = 0; g < RPW; ++g) {
            const int t = __ffs(rows) - 1;
            rows &= rows - 1;
            if (g == seg) b = t;
        }
        const int64_t at = __shfl_sync(0xffffffffu, p0, b & 31);
        L = __shfl_sync(0xffffffffu, len, b & 31);
        if (b < 0) L = 0;
        c = -1;
        a = 0.f;
        if (sl < L) {
            c = ld_once(col + at + sl);
            a = ld_once(val + at + sl);
        }
    };
    fetch();
    for (bool more = true; more;) {
        const int rb = b, Lc = L;
        const bool in = (unsigned)c < (unsigned)d;
        const int cp = in ? c : -1;
        const float ap = in ? a : 0.f;
        more = rows != 0;
        if (more) fetch();
        const int half = Lc >> 1;
        // steps this lane takes: the last one of an even length belongs to the lower half of the lanes
        const int mine = !in ? 0 : ((Lc & 1) == 0 && sl >= half ? half - 1 : half);
        const int steps = RPW > 1 ? (int)__reduce_max_sync(0xffffffffu, (unsigned)half) : half;
        const float2* Prow = P + (in ? cp * d : 0);
        const f32x2 a2 = pack2(ap, ap);
        f32x2 sh = 0ull, se = 0ull;
        for (int s0 = 1; s0 <= steps; s0 += 4) {
            float2 Pq[4];
            float aq[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                int t = sl + s0 + u;
                t -= t >= Lc ? Lc : 0;
                const int src = lane - sl + (t & (SEG - 1));
                const int cq = __shfl_sync(0xffffffffu, cp, src);
                const float x = __shfl_sync(0xffffffffu, ap, src);
                const bool ok = s0 + u <= mine && cq >= 0;
                Pq[u] = make_float2(0.f, 0.f);
                if (ok) Pq[u] = __ldg(Prow + cq);
                aq[u] = ok ? x : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; u += 2) {
                const f32x2 q = pack2(aq[u], aq[u + 1]);
                const f32x2 hi = pack2(Pq[u].x, Pq[u + 1].x), lo = pack2(Pq[u].y, Pq[u + 1].y);
                const f32x2 x = mul2(a2, q);
                const f32x2 xe = fma2(a2, q, neg2(x));                // a_p a_q = x + xe exactly
                const f32x2 th = mul2(x, hi);
                f32x2 tl = fma2(x, hi, neg2(th));
                tl = fma2(x, lo, tl);
                tl = fma2(xe, hi, tl);
                const f32x2 sum = add2(sh, th);                       // TwoSum; the remainders collect in se
                const f32x2 bb = sub2(sum, sh);
                const f32x2 er = add2(sub2(sh, sub2(sum, bb)), sub2(th, bb));
                se = add2(se, add2(er, tl));
                sh = sum;
            }
        }
        float h0, h1, e0, e1;
        unpack2(sh, h0, h1);
        unpack2(se, e0, e1);
        df_add(h0, e0, h1, e1);
        h0 = __fmul_rn(h0, 2.f);
        e0 = __fmul_rn(e0, 2.f);
        float dh = 0.f, dl = 0.f;
        if (in) df_term(ap, ap, 1.f, dg[cp], dh, dl);
        df_add(h0, e0, dh, dl);
#pragma unroll
        for (int o = SEG / 2; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, h0, o), oe = __shfl_xor_sync(0xffffffffu, e0, o);
            df_add(h0, e0, oh, oe);
        }
        if (sl == 0 && rb >= 0) theta[r0 + rb] = __fadd_rn(h0, e0);
    }
}

// Every row of at most 32 entries by the second form (an empty row gets 0): a warp reads the bounds of 32 rows
// at once (the next 32 loaded ahead), takes them by class, 8, 16 or 32 lanes a row, and notes whether any is
// longer. Bound by L1 at 89%: each
// read of P is a line of its own (P is 8 MB at d = 1,024, 2% of the reads hit), so len (len - 1) / 2 reads a row
// with the diagonal in shared memory instead of len (len + 1) / 2, and one pass over the bounds instead of one
// for each class, are what counts. 8e7 rows of 12 entries, d = 1,024: 29.3 -> 19.5 ms with k_final_csr_long
// (a lane took the pairs (p, q >= p), one read in flight a warp); 8e6 rows of 8 with 1% of 256: 2.9 -> 2.1 ms.
__global__ void __launch_bounds__(256) k_final_csr_pairs(const int64_t* __restrict__ row_ptr,
                                                         const int32_t* __restrict__ col,
                                                         const float* __restrict__ val, int64_t n, int d,
                                                         const float2* __restrict__ P, int* __restrict__ longer_seen,
                                                         float* __restrict__ theta) {
    __shared__ float2 dg[1024];
    for (int j = threadIdx.x; j < d; j += blockDim.x) dg[j] = P[(int64_t)j * (d + 1)];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int64_t rn = warp * 32 + lane;
    int64_t np0 = rn < n ? row_ptr[rn] : 0, np1 = rn < n ? row_ptr[rn + 1] : -1;
    for (int64_t r0 = warp * 32; r0 < n; r0 += nwarps * 32) {
        const int64_t p0 = np0, len64 = np1 - np0;                    // past the end: length -1, in no class
        rn += nwarps * 32;
        np0 = rn < n ? row_ptr[rn] : 0;
        np1 = rn < n ? row_ptr[rn + 1] : -1;
        const int len = (int)min(len64, (int64_t)64);
        const unsigned m8 = __ballot_sync(0xffffffffu, len64 >= 0 && len64 <= 8);
        const unsigned m16 = __ballot_sync(0xffffffffu, len64 > 8 && len64 <= 16);
        const unsigned m32 = __ballot_sync(0xffffffffu, len64 > 16 && len64 <= 32);
        if (__any_sync(0xffffffffu, len64 > 32) && lane == 0) *longer_seen = 1;
        csr_pair_rows<8>(m8, p0, len, r0, lane, col, val, d, P, dg, theta);
        csr_pair_rows<16>(m16, p0, len, r0, lane, col, val, d, P, dg, theta);
        csr_pair_rows<32>(m32, p0, len, r0, lane, col, val, d, P, dg, theta);
    }
}

// Rows of more than 32 entries by the first form: a warp scans the bounds of 32 rows at once (the next 32
// loaded ahead) and takes each such row in turn; nothing to do when k_final_csr_pairs saw no such row (the scan
// alone took 0.46 ms at 8e7 rows). Finding the rows by masks that the pairs' pass leaves, or scanning 128 bounds
// at once, cost registers that the rows' own loop needs (1.46 against 1.30 ms at 8e4 rows of 256 entries).
template <bool VEC>
__global__ void __launch_bounds__(256) k_final_csr_long(const int64_t* __restrict__ row_ptr,
                                                        const int32_t* __restrict__ col,
                                                        const float* __restrict__ val, int64_t n, int d,
                                                        const float* __restrict__ M, int k,
                                                        const int* __restrict__ seen, float* __restrict__ theta) {
    if (!*seen) return;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int64_t rn = warp * 32 + lane;
    int64_t np0 = rn < n ? row_ptr[rn] : 0, np1 = rn < n ? row_ptr[rn + 1] : 0;
    for (int64_t r0 = warp * 32; r0 < n; r0 += nwarps * 32) {
        const int64_t b0 = np0, b1 = np1;
        rn += nwarps * 32;
        np0 = rn < n ? row_ptr[rn] : 0;
        np1 = rn < n ? row_ptr[rn + 1] : 0;
        unsigned todo = __ballot_sync(0xffffffffu, b1 - b0 > 32);
        while (todo) {
            const int b = __ffs(todo) - 1;
            todo &= todo - 1;
            const int64_t p0 = __shfl_sync(0xffffffffu, b0, b), p1 = __shfl_sync(0xffffffffu, b1, b);
            const float total = warp_sum(csr_row_norm<VEC>(p0, p1, col, val, d, M, k, lane));
            if (lane == 0) theta[r0 + b] = total;
        }
    }
}

// Pdf (d x d pairs) = P split into FP32 hi + lo.
__global__ void k_split_pairs(const double* __restrict__ P, int64_t count, float2* __restrict__ Pdf) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x) {
        const double x = P[e];
        const float h = (float)x;
        Pdf[e] = make_float2(h, (float)(x - (double)h));
    }
}

// MT (k x d) = Mfull^T (Mfull d x k, both row-major).
__global__ void k_transpose_mfull(const float* __restrict__ M, int d, int k, float* __restrict__ MT) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)d * k;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int q = (int)(e / d), c = (int)(e % d);
        MT[e] = M[(int64_t)c * k + q];
    }
}

}  // namespace

cudaError_t launch_final_dense_fp32(const float* A, int64_t lda, int64_t n, int64_t d,
                                    const float* Mfull, int64_t k, float* theta, cudaStream_t st) {
    const bool vec = (reinterpret_cast<uintptr_t>(A) % 16 == 0) && (reinterpret_cast<uintptr_t>(Mfull) % 16 == 0) &&
                     (lda % 4 == 0) && (d % 4 == 0) && (k % 4 == 0);
    // 128 rows a CTA, one CTA an SM; below two rounds of them, 64 rows and two CTAs an SM
    const bool big = n >= 2 * 152 * 128;
    const int64_t bm = big ? 128 : 64, grid = (n + bm - 1) / bm;
    if (grid > 0x7fffffff) return cudaErrorInvalidValue;
    const unsigned g = (unsigned)grid;
    if (vec && big)
        k_final_dense_fp32<true, 8><<<g, 256, 0, st>>>(A, lda, n, (int)d, Mfull, (int)k, theta);
    else if (vec)
        k_final_dense_fp32<true, 4><<<g, 256, 0, st>>>(A, lda, n, (int)d, Mfull, (int)k, theta);
    else if (big)
        k_final_dense_fp32<false, 8><<<g, 256, 0, st>>>(A, lda, n, (int)d, Mfull, (int)k, theta);
    else
        k_final_dense_fp32<false, 4><<<g, 256, 0, st>>>(A, lda, n, (int)d, Mfull, (int)k, theta);
    return cudaGetLastError();
}

size_t csr_gram_scratch_bytes(int64_t d, int64_t k) {
    return sizeof(double) * (size_t)(d * d + gram_partial_doubles(k, d)) + sizeof(float) * (size_t)(k * d) +
           sizeof(float2) * (size_t)(d * d) + 1024;
}

bool csr_gram_pays(int64_t n, int64_t d, int64_t nnz, int64_t k) {
    return d <= 1024 && n > 0 && nnz * 8 < n * k;      // short rows on average: nnz_i < k / 8
}

cudaError_t launch_final_csr_gram(const int64_t* row_ptr, const int32_t* col, const float* val, int64_t n, int64_t d,
                                  const float* Mfull, int64_t k, void* scratch, float* theta, int32_t* status,
                                 cudaStream_t st) {
    double* P = reinterpret_cast<double*>(scratch);
    double* Gp = P + d * d;
    float* MT = reinterpret_cast<float*>(Gp + gram_partial_doubles(k, d));
    float2* Pdf = reinterpret_cast<float2*>(reinterpret_cast<uintptr_t>(MT + k * d + 3) & ~uintptr_t(7));
    int* seen = reinterpret_cast<int*>(Pdf + d * d);    // a row of more than 32 entries was met
    cudaError_t e = cudaMemsetAsync(seen, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    int tg = (int)((d * k + 255) / 256);
    if (tg > 152 * 8) tg = 152 * 8;
    k_transpose_mfull<<<tg, 256, 0, st>>>(Mfull, (int)d, (int)k, MT);
    e = launch_gram_fp64(MT, d, k, d, Gp, P, status, st);           // P = Mfull Mfull^T (FP64-grade)
    if (e != cudaSuccess) return e;
    k_split_pairs<<<152 * 4, 256, 0, st>>>(P, d * d, Pdf);
    const bool vec = (reinterpret_cast<uintptr_t>(Mfull) % 16 == 0) && (k % 4 == 0);
    int64_t grid = (n + 255) / 256;                     // 32 rows a warp at a time
    if (grid > 152 * 24) grid = 152 * 24;
    if (grid < 1) grid = 1;
    k_final_csr_pairs<<<(unsigned)grid, 256, 0, st>>>(row_ptr, col, val, n, (int)d, Pdf, seen, theta);  // empty rows too
    int64_t grid_l = (n + 255) / 256;                   // 32 rows scanned a warp
    if (grid_l > 152 * 16) grid_l = 152 * 16;
    if (grid_l < 1) grid_l = 1;
    if (vec)
        k_final_csr_long<true><<<(unsigned)grid_l, 256, 0, st>>>(row_ptr, col, val, n, (int)d, Mfull, (int)k, seen,
                                                                theta);
    else
        k_final_csr_long<false><<<(unsigned)grid_l, 256, 0, st>>>(row_ptr, col, val, n, (int)d, Mfull, (int)k, seen,
                                                                 theta);
    return cudaGetLastError();
}

cudaError_t launch_final_csr_fp32(const int64_t* row_ptr, const int32_t* col, const float* val,
                                  int64_t n, int64_t d, const float* Mfull, int64_t k,
                                  float* theta, cudaStream_t st) {
    const bool vec = (reinterpret_cast<uintptr_t>(Mfull) % 16 == 0) && (k % 4 == 0);
    int64_t grid = (n * 32 + 255) / 256;
    if (grid > 152 * 64) grid = 152 * 64;
    if (grid < 1) grid = 1;
    if (vec)
        k_final_csr_fp32<true><<<(unsigned)grid, 256, 0, st>>>(row_ptr, col, val, n, (int)d, Mfull, (int)k, theta);
    else
        k_final_csr_fp32<false><<<(unsigned)grid, 256, 0, st>>>(row_ptr, col, val, n, (int)d, Mfull, (int)k, theta);
    return cudaGetLastError();
}

}  // namespace lev
