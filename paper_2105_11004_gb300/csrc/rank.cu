// Rank decisions beyond the diagonal test of the pivoted QR, on sm_103a (FP64).
//
//  * singular values of the sketch: one-sided (Hestenes) Jacobi on the rows of R, the triangular
//    factor of A~ P (sigma(R) = sigma(A~)): plane rotations of row pairs (Y <- J Y) until every
//    pair is orthogonal, after which the row norms are the singular values and the normalised rows
//    the right singular vectors of R. One thread-block cluster with the rows in shared memory up to
//    d = 384, one cooperative grid above (the pairs of a round are disjoint, round-robin order). The rank is then the count
//    of sigma_j > tau sigma_1 (Alg. 11 step 3; Sec. 7.2: the singular values see a gap that the
//    diagonal of R can miss);
//  * strong-RRQR measures at a fixed k (Alg. 2 after Gu and Eisenstat): from R in pivot order,
//    Z = R11^{-1} [I | R12], the row norms of R11^{-1}, gamma_j^2 = G_jj - ||R[:k, j]||^2 (the
//    Schur complement's diagonal, G = A~^T A~), and the largest
//    rho_ij^2 = (R11^{-1} R12)_ij^2 + gamma_j^2 ||e_i^T R11^{-1}||^2 with its (i, j).
#include <atomic>

#include "df.cuh"
#include "f32x2.cuh"
#include "lev_common.cuh"
#include "lev_kernels.cuh"

namespace lev {

namespace {

constexpr double kJacobiTol = 1e-12;   // a pair counts as orthogonal when |y_p.y_q| <= tol ||y_p|| ||y_q||

__device__ __forceinline__ void round_pair(int n, int t, int i, int& p, int& q) {
    if (i == 0) {
        p = t;
        q = n - 1;
    } else {
        p = (t + i) % (n - 1);
        q = (t - i + n - 1) % (n - 1);
    }
}

__device__ __forceinline__ void st_release_gpu(unsigned* p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

// Double-float arithmetic (a value is hi + lo, two FP32 numbers, about 48 significant bits): FP64
// runs at 1/64 of the FP32 rate on this GPU, and the Jacobi's dot products and rotations are its
// bulk. Every step uses the round-to-nearest intrinsics, so nothing is contracted into an FMA that
// would break the error-free transformations (Knuth's TwoSum, the fma-based TwoProduct).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ void df_add(float ah, float al, float bh, float bl, float& sh, float& sl) {
    float s, e;
    two_sum(ah, bh, s, e);
    e = __fadd_rn(e, __fadd_rn(al, bl));
    two_sum(s, e, sh, sl);
}

// (ah + al)(bh + bl), the al bl term dropped (below 2^-48 of the product)
__device__ __forceinline__ void df_mul(float ah, float al, float bh, float bl, float& ph, float& pl) {
    const float p = __fmul_rn(ah, bh);
    float e = __fmaf_rn(ah, bh, -p);
    e = __fmaf_rn(ah, bl, e);
    e = __fmaf_rn(al, bh, e);
    two_sum(p, e, ph, pl);
}

// (s, c) += (xh + xl)(yh + yl): the exact product xh yh = p + e, the cross terms into e, p added
// error-free to s, the errors collected in c
__device__ __forceinline__ void df_dot_acc(float xh, float xl, float yh, float yl, float& s, float& c) {
    const float p = __fmul_rn(xh, yh);
    float e = __fmaf_rn(xh, yh, -p);
    e = __fmaf_rn(xh, yl, e);
    e = __fmaf_rn(xl, yh, e);
    float s1, q;
    two_sum(s, p, s1, q);
    s = s1;
    c = __fadd_rn(c, __fadd_rn(q, e));
}

// the same pair on every lane (df_add is symmetric in its two arguments)
__device__ __forceinline__ void df_warp_sum(float& h, float& l) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
        df_add(h, l, oh, ol, h, l);
    }
}

// Yh, Yl = the double-float split of R (hi = fl32(x), lo = fl32(x - hi)); Y = Yh + Yl back in FP64.
__global__ void k_split_rows(const double* __restrict__ R, int64_t count, float* __restrict__ Yh,
                             float* __restrict__ Yl) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x) {
        const double x = R[e];
        const float h = (float)x;
        Yh[e] = h;
        Yl[e] = (float)(x - (double)h);
    }
}

__global__ void k_join_rows(const float* __restrict__ Yh, const float* __restrict__ Yl, int64_t count,
                            double* __restrict__ Y) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        Y[e] = (double)Yh[e] + (double)Yl[e];
}

// One-sided Jacobi on rows 0..r-1 (r read from *d_rows, at most d) of Y = Yh + Yl (double-float,
// row-major, ld = d), one CTA a pair: thread t holds elements t + 256 j (j < PER, d <= 256 PER) of
// both rows; the three dot products are compensated sums reduced over the warps in double-float
// and over the CTA in FP64 by one thread, which also takes the rotation (in FP64) and splits it;
// the rotation itself runs in double-float. Rounds are ordered by rows, not by a grid barrier:
// version[p] (zeroed by the caller) counts the rounds applied to row p, and the CTA that holds pair
// (p, q) in global round T waits (bounded) until both rows reached version T, rotates them and
// publishes T + 1. Every CTA takes its pairs in round order and all CTAs are resident (cooperative
// launch), so the earliest unfinished pair always has its rows ready. A grid barrier ends each
// sweep; rotated[s] counts the rotations of sweep s (zeroed by the caller) and the sweeps stop
// after one without any. *sweeps_out = sweeps run (max_sweeps + 1 when the last sweep still
// rotated).
template <int PER>
__global__ void __launch_bounds__(256) k_jacobi_rows(float* __restrict__ Yh, float* __restrict__ Yl,
                                                     const int64_t* __restrict__ d_rows, int d, int max_sweeps,
                                                     unsigned* __restrict__ rotated, unsigned* __restrict__ barrier,
                                                     unsigned* __restrict__ version, int32_t* __restrict__ status,
                                                     int32_t* __restrict__ sweeps_out) {
    __shared__ float part[6][8];
    __shared__ float rot[4];
    __shared__ int do_rot;
    const int r = (int)min(max(*d_rows, (int64_t)0), (int64_t)d);
    const int n = r + (r & 1);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    unsigned epoch = 0;
    if (n < 2) {
        if (blockIdx.x == 0 && tid == 0) *sweeps_out = 0;
        return;
    }
    for (int s = 0; s < max_sweeps; ++s) {
        for (int t = 0; t < n - 1; ++t) {
            const unsigned T = (unsigned)s * (unsigned)(n - 1) + (unsigned)t;
            for (int i = blockIdx.x; i < n / 2; i += gridDim.x) {
                int p, q;
                round_pair(n, t, i, p, q);
                const bool pv = p < r, qv = q < r;                       // q may be the padding row
                if (tid == 0) {
                    long long spins = 0;
                    while ((pv && ld_acquire_gpu(version + p) < T) || (qv && ld_acquire_gpu(version + q) < T)) {
                        if (ld_volatile(status) != 0) break;
                        if (++spins > kSpinLimit) {
                            atomicExch(status, kStatusTimeoutBarrier);
                            break;
                        }
                        __nanosleep(32);
                    }
                }
                __syncthreads();
                if (ld_volatile(status) != 0) return;
                if (pv && qv) {
                    float xh[PER], xl[PER], yh[PER], yl[PER];
                    const int64_t op = (int64_t)p * d, oq = (int64_t)q * d;
#pragma unroll
                    for (int j = 0; j < PER; ++j) {
                        const int e = tid + 256 * j;
                        const bool ok = e < d;
                        xh[j] = ok ? Yh[op + e] : 0.f;
                        xl[j] = ok ? Yl[op + e] : 0.f;
                        yh[j] = ok ? Yh[oq + e] : 0.f;
                        yl[j] = ok ? Yl[oq + e] : 0.f;
                    }
                    float ah = 0.f, al = 0.f, bh = 0.f, bl = 0.f, ch = 0.f, cl = 0.f;
#pragma unroll
                    for (int j = 0; j < PER; ++j) {
                        df_dot_acc(xh[j], xl[j], xh[j], xl[j], ah, al);
                        df_dot_acc(yh[j], yl[j], yh[j], yl[j], bh, bl);
                        df_dot_acc(xh[j], xl[j], yh[j], yl[j], ch, cl);
                    }
                    df_warp_sum(ah, al);
                    df_warp_sum(bh, bl);
                    df_warp_sum(ch, cl);
                    if (lane == 0) {
                        part[0][w] = ah; part[1][w] = al;
                        part[2][w] = bh; part[3][w] = bl;
                        part[4][w] = ch; part[5][w] = cl;
                    }
                    __syncthreads();
                    if (tid == 0) {
                        double a = 0.0, b = 0.0, c = 0.0;
                        for (int u = 0; u < 8; ++u) {
                            a += (double)part[0][u] + (double)part[1][u];
                            b += (double)part[2][u] + (double)part[3][u];
                            c += (double)part[4][u] + (double)part[5][u];
                        }
                        int go = 0;
                        if (a > 0.0 && b > 0.0 && fabs(c) > kJacobiTol * sqrt(a) * sqrt(b)) {
                            const double zeta = (b - a) / (2.0 * c);
                            const double tr = copysign(1.0, zeta) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                            const double cs = 1.0 / sqrt(1.0 + tr * tr), sn = cs * tr;
                            const float csh = (float)cs, snh = (float)sn;
                            rot[0] = csh;
                            rot[1] = (float)(cs - (double)csh);
                            rot[2] = snh;
                            rot[3] = (float)(sn - (double)snh);
                            go = 1;
                            atomicAdd(&rotated[s], 1u);
                        }
                        do_rot = go;
                    }
                    __syncthreads();
                    if (do_rot) {
                        const float csh = rot[0], csl = rot[1], snh = rot[2], snl = rot[3];
#pragma unroll
                        for (int j = 0; j < PER; ++j) {
                            const int e = tid + 256 * j;
                            if (e >= d) continue;
                            float t1h, t1l, t2h, t2l, nh, nl;
                            df_mul(csh, csl, xh[j], xl[j], t1h, t1l);             // x' = cs x - sn y
                            df_mul(snh, snl, yh[j], yl[j], t2h, t2l);
                            df_add(t1h, t1l, -t2h, -t2l, nh, nl);
                            Yh[op + e] = nh;
                            Yl[op + e] = nl;
                            df_mul(snh, snl, xh[j], xl[j], t1h, t1l);             // y' = sn x + cs y
                            df_mul(csh, csl, yh[j], yl[j], t2h, t2l);
                            df_add(t1h, t1l, t2h, t2l, nh, nl);
                            Yh[oq + e] = nh;
                            Yl[oq + e] = nl;
                        }
                    }
                }
                __syncthreads();                                             // rows written, rot read
                if (tid == 0) {
                    __threadfence();
                    if (pv) st_release_gpu(version + p, T + 1);
                    if (qv) st_release_gpu(version + q, T + 1);
                }
            }
        }
        if (!grid_barrier(barrier, epoch, status)) return;
        if (*(volatile unsigned*)&rotated[s] == 0u) {
            if (blockIdx.x == 0 && tid == 0) *sweeps_out = s + 1;
            return;
        }
    }
    if (blockIdx.x == 0 && tid == 0) *sweeps_out = max_sweeps + 1;
}

// ---- the same Jacobi on one thread-block cluster, the rows in shared memory (d up to about 400) ----
// k_jacobi_rows spends a round on L2: two row versions polled, two rows read, written and released, about
// 7.5 us for one pair a CTA, whatever the arithmetic. Here the r rows are cut into 2 C blocks of b rows, two
// blocks a CTA (C = 1 .. 16 CTAs, b = 8 at d = 256), and a sweep is 2 C - 1 block rounds of the round-robin
// tournament: a CTA takes the b x b pairs between its two blocks in b steps of b disjoint pairs, a warp a
// pair, and the blocks then move on through distributed shared memory (each CTA pulls its next two blocks
// into its other buffer; one cluster barrier a block round). The pairs inside the blocks come first. A warp
// keeps its row of the first block in registers through the b steps. The squared row norms are carried
// (recomputed every sweep), so a pair costs one dot product; the rotation's tangent is taken in FP32 (its
// error of 1e-7 leaves 1e-7 of the pair's dot product to the next sweep) and made a rotation in double-float,
// c = 1 / sqrt(1 + t^2), s = c t, which is what keeps the rows' accuracy. Two elements an instruction
// (packed FP32). Same stopping rule as k_jacobi_rows; singular values at d = 256: 5.7e-14 off (8.8e-14 there).
// The SVD path with its QR: 24.1 -> 6.5 ms at 1,024 x 256 (Jacobi 21.5 -> 3.4), 7.9 -> 1.8 at d = 99, 45.4 -> 15.6
// at d = 384. A pair is a chain of about 2,500 cycles: dot product and its warp sum, rotation, update, barrier.
// A row held by a warp: lane l has elements 128 q + 4 l .. + 3, as 2 Q packed pairs of high and low parts.
template <int Q>
struct JRow {
    f32x2 h[2 * Q], l[2 * Q];
};
template <int Q>
__device__ __forceinline__ void load_row(const float* row, int dp, int lane, JRow<Q>& v) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(row + 128 * q + 4 * lane);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(row + dp + 128 * q + 4 * lane);
        v.h[2 * q] = a.x; v.h[2 * q + 1] = a.y;
        v.l[2 * q] = b.x; v.l[2 * q + 1] = b.y;
    }
}
template <int Q>
__device__ __forceinline__ void store_row(float* row, int dp, int lane, const JRow<Q>& v) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        *reinterpret_cast<ulonglong2*>(row + 128 * q + 4 * lane) = make_ulonglong2(v.h[2 * q], v.h[2 * q + 1]);
        *reinterpret_cast<ulonglong2*>(row + dp + 128 * q + 4 * lane) = make_ulonglong2(v.l[2 * q], v.l[2 * q + 1]);
    }
}
// x . y over the warp (the same pair on every lane): compensated as df_dot_acc, two elements at a time
template <int Q>
__device__ __forceinline__ float2 row_dot(const JRow<Q>& x, const JRow<Q>& y) {
    f32x2 s = 0ull, c = 0ull;
#pragma unroll
    for (int k = 0; k < 2 * Q; ++k) {
        const f32x2 p = mul2(x.h[k], y.h[k]);
        f32x2 e = fma2(x.h[k], y.h[k], neg2(p));
        e = fma2(x.h[k], y.l[k], e);
        e = fma2(x.l[k], y.h[k], e);
        const f32x2 s1 = add2(s, p), z = sub2(s1, s);
        c = add2(c, add2(add2(sub2(s, sub2(s1, z)), sub2(p, z)), e));
        s = s1;
    }
    float s0, s1, c0, c1, h, l;
    unpack2(s, s0, s1);
    unpack2(c, c0, c1);
    df_add(s0, c0, s1, c1, h, l);
    df_warp_sum(h, l);
    return make_float2(h, l);
}
// (ah + al) u + (bh + bl) v for packed double-float u, v and scalars broadcast to both halves
__device__ __forceinline__ void df_axpby(f32x2 ah, f32x2 al, f32x2 uh, f32x2 ul, f32x2 bh, f32x2 bl, f32x2 vh, f32x2 vl,
                                         f32x2& oh, f32x2& ol) {
    const f32x2 p = mul2(ah, uh), q = mul2(bh, vh);
    f32x2 e = fma2(ah, uh, neg2(p)), f = fma2(bh, vh, neg2(q));
    e = fma2(ah, ul, e);
    f = fma2(bh, vl, f);
    e = fma2(al, uh, e);
    f = fma2(bl, vh, f);
    const f32x2 s = add2(p, q), z = sub2(s, p);
    f32x2 r = add2(sub2(p, sub2(s, z)), sub2(q, z));
    r = add2(r, add2(e, f));
    oh = add2(s, r);
    ol = sub2(r, sub2(oh, s));
}
// 1 / sqrt(v) for v = vh + vl in [1, 2]: an FP32 estimate y with residual e = 1 - v y^2 (about 2^-23; its leading
// difference is exact), then y (1 + e / 2 + 3 e^2 / 8).
__device__ __forceinline__ float2 inv_sqrt_1to2(float vh, float vl) {
    float y = rsqrtf(vh);
    y = __fmul_rn(y, __fmaf_rn(__fmul_rn(-0.5f, vh), __fmul_rn(y, y), 1.5f));
    const float yy = __fmul_rn(y, y), yye = __fmaf_rn(y, y, -yy);
    const float p = __fmul_rn(vh, yy), pe = __fmaf_rn(vh, yy, -p);
    const float e = __fsub_rn(__fsub_rn(1.f, p), __fadd_rn(pe, __fmaf_rn(vh, yye, __fmul_rn(vl, yy))));
    const float corr = __fmul_rn(y, __fmul_rn(e, __fmaf_rn(0.375f, e, 0.5f)));
    const float h = __fadd_rn(y, corr);
    return make_float2(h, __fsub_rn(corr, __fsub_rn(h, y)));
}
// The pair (cs, sn) made orthonormal to a few 2^-50: the residual 1 - cs^2 - sn^2 (its leading differences are
// exact, the other terms summed error-free) goes half into each low part. An error here scales both rows at
// every rotation; the FP64 rotations of k_jacobi_rows, split into pairs, have the same 8e-16.
__device__ __forceinline__ void orthonormalise(float2& cs, float2& sn) {
    const float p1 = __fmul_rn(cs.x, cs.x), e1 = __fmaf_rn(cs.x, cs.x, -p1);
    const float p2 = __fmul_rn(sn.x, sn.x), e2 = __fmaf_rn(sn.x, sn.x, -p2);
    const float c2 = 2.f * cs.x, s2 = 2.f * sn.x;
    const float m1 = __fmul_rn(c2, cs.y), n1 = __fmaf_rn(c2, cs.y, -m1);
    const float m2 = __fmul_rn(s2, sn.y), n2 = __fmaf_rn(s2, sn.y, -m2);
    float s = __fsub_rn(__fsub_rn(1.f, p1), p2), a, b, c, d;
    two_sum(s, -e1, s, a);
    two_sum(s, -e2, s, b);
    two_sum(s, -m1, s, c);
    two_sum(s, -m2, s, d);
    const float low = __fsub_rn(__fadd_rn(__fadd_rn(a, b), __fadd_rn(c, d)),
                                __fadd_rn(__fadd_rn(n1, n2), __fmaf_rn(cs.y, cs.y, __fmul_rn(sn.y, sn.y))));
    const float half = 0.5f * __fadd_rn(s, low);
    cs.y = __fmaf_rn(cs.x, half, cs.y);
    sn.y = __fmaf_rn(sn.x, half, sn.y);
}
// Rotate rows x, y (squared norms a, b) so that they become orthogonal; false if they count as orthogonal.
template <int Q>
__device__ __forceinline__ bool rotate_rows(JRow<Q>& x, JRow<Q>& y, float2& a, float2& b) {
    const float2 c = row_dot<Q>(x, y);
    if (!(a.x > 0.f && b.x > 0.f && fabsf(c.x) > (float)kJacobiTol * sqrtf(a.x) * sqrtf(b.x))) return false;
    const float zeta = ((b.x - a.x) + (b.y - a.y)) / (2.f * c.x);
    const float az = fabsf(zeta);
    const float t = copysignf(az > 1e9f ? 0.5f / az : 1.f / (az + sqrtf(fmaf(az, az, 1.f))), zeta);
    const float tt = __fmul_rn(t, t), tte = __fmaf_rn(t, t, -tt);
    const float vh = __fadd_rn(1.f, tt);
    const float vl = __fadd_rn(__fsub_rn(tt, __fsub_rn(vh, 1.f)), tte);                 // 1 + t^2 (t^2 <= 1)
    float2 cs = inv_sqrt_1to2(vh, vl), sn = lev::df_mul(cs, make_float2(t, 0.f));
    orthonormalise(cs, sn);
    const f32x2 ch = pack2(cs.x, cs.x), cl = pack2(cs.y, cs.y), sh = pack2(sn.x, sn.x), sl = pack2(sn.y, sn.y);
    const f32x2 nsh = pack2(-sn.x, -sn.x), nsl = pack2(-sn.y, -sn.y);
#pragma unroll
    for (int k = 0; k < 2 * Q; ++k) {
        f32x2 xh, xl;
        df_axpby(ch, cl, x.h[k], x.l[k], nsh, nsl, y.h[k], y.l[k], xh, xl);             // x' = cs x - sn y
        df_axpby(sh, sl, x.h[k], x.l[k], ch, cl, y.h[k], y.l[k], y.h[k], y.l[k]);       // y' = sn x + cs y
        x.h[k] = xh;
        x.l[k] = xl;
    }
    const float2 tc = lev::df_mul(c, make_float2(t, 0.f));
    float h, l;
    df_add(a.x, a.y, -tc.x, -tc.y, h, l);
    a = make_float2(h, l);
    df_add(b.x, b.y, tc.x, tc.y, h, l);
    b = make_float2(h, l);
    return true;
}

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t remote_addr(const void* p, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ uint4 remote_ld16(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}

constexpr int kJacobiMaxWarps = 16;

// bmax: rows a block holds at most (warps of the CTA); dp = 128 Q >= d. Dynamic shared memory: two buffers of
// two blocks of bmax rows of 2 dp floats (high parts, low parts).
template <int Q>
__global__ void __launch_bounds__(32 * kJacobiMaxWarps, 1) k_jacobi_cluster(float* __restrict__ Yh, float* __restrict__ Yl,
                                                                           const int64_t* __restrict__ d_rows, int d,
                                                                           int bmax, int max_sweeps,
                                                                           int32_t* __restrict__ sweeps_out) {
    constexpr int dp = 128 * Q;
    extern __shared__ __align__(16) float jrows[];
    __shared__ __align__(16) float2 norm_s[2][2][kJacobiMaxWarps];   // by buffer and block: squared norms
    __shared__ __align__(16) int id_s[2][2][kJacobiMaxWarps];        // rows of Y held (-1: none)
    __shared__ int rotated_s[2];
    uint32_t C, me;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(me));
    const int r = (int)min(max(*d_rows, (int64_t)0), (int64_t)d);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int b = (r + 2 * (int)C - 1) / (2 * (int)C);
    if (r < 2) {                                            // the same in every CTA
        if (me == 0 && threadIdx.x == 0) *sweeps_out = 0;
        return;
    }
    auto row = [&](int buf, int blk, int i) -> float* { return jrows + ((size_t)(buf * 2 + blk) * bmax + i) * (2 * dp); };
    // blocks 2 me and 2 me + 1
    for (int blk = 0; blk < 2; ++blk)
        for (int i = w; i < b; i += nw) {
            const int id = (2 * (int)me + blk) * b + i;
            float* dst = row(0, blk, i);
            for (int e = lane; e < dp; e += 32) {
                const bool ok = id < r && e < d;
                dst[e] = ok ? Yh[(int64_t)id * d + e] : 0.f;
                dst[dp + e] = ok ? Yl[(int64_t)id * d + e] : 0.f;
            }
            if (lane == 0) id_s[0][blk][i] = id < r ? id : -1;
        }
    if (threadIdx.x < 2) rotated_s[threadIdx.x] = 0;
    __syncthreads();
    int buf = 0, sweep = 0;
    const int rounds = 2 * (int)C - 1;
    for (; sweep < max_sweeps; ++sweep) {
        int rotations = 0;                                 // by this warp (lane 0's count)
        // squared norms afresh
        for (int i = w; i < 2 * b; i += nw) {
            JRow<Q> x;
            load_row<Q>(row(buf, i / b, i % b), dp, lane, x);
            const float2 n2 = row_dot<Q>(x, x);
            if (lane == 0) norm_s[buf][i / b][i % b] = n2;
        }
        __syncthreads();
        // the pairs inside the two blocks
        const int n = b + (b & 1);
        for (int t = 0; t < n - 1; ++t) {
            for (int e = w; e < n; e += nw) {                // n / 2 pairs a block
                const int blk = e / (n / 2);
                int p, q;
                round_pair(n, t, e % (n / 2), p, q);
                if (p >= b || q >= b || id_s[buf][blk][p] < 0 || id_s[buf][blk][q] < 0) continue;
                if (p > q) { const int x = p; p = q; q = x; }
                JRow<Q> x, y;
                load_row<Q>(row(buf, blk, p), dp, lane, x);
                load_row<Q>(row(buf, blk, q), dp, lane, y);
                float2 na = norm_s[buf][blk][p], nb = norm_s[buf][blk][q];
                if (rotate_rows<Q>(x, y, na, nb)) {
                    store_row<Q>(row(buf, blk, p), dp, lane, x);
                    store_row<Q>(row(buf, blk, q), dp, lane, y);
                    if (lane == 0) { norm_s[buf][blk][p] = na; norm_s[buf][blk][q] = nb; }
                    ++rotations;
                }
            }
            __syncthreads();
        }
        for (int rd = 0; rd < rounds; ++rd) {
            // warp w holds row w of the first block; step k pairs it with row (w + k) mod b of the second
            const bool mine = w < b && id_s[buf][0][w] >= 0;
            JRow<Q> x;
            float2 na = make_float2(0.f, 0.f);
            bool changed = false;
            if (mine) {
                load_row<Q>(row(buf, 0, w), dp, lane, x);
                na = norm_s[buf][0][w];
            }
            for (int k = 0; k < b; ++k) {
                if (mine) {
                    const int j = w + k < b ? w + k : w + k - b;
                    if (id_s[buf][1][j] >= 0) {
                        JRow<Q> y;
                        load_row<Q>(row(buf, 1, j), dp, lane, y);
                        float2 nb = norm_s[buf][1][j];
                        if (rotate_rows<Q>(x, y, na, nb)) {
                            store_row<Q>(row(buf, 1, j), dp, lane, y);
                            if (lane == 0) norm_s[buf][1][j] = nb;
                            changed = true;
                            ++rotations;
                        }
                    }
                }
                __syncthreads();
            }
            if (changed) {
                store_row<Q>(row(buf, 0, w), dp, lane, x);
                if (lane == 0) norm_s[buf][0][w] = na;
            }
            if (rd == rounds - 1 && lane == 0 && rotations) atomicAdd(&rotated_s[sweep & 1], rotations);
            if (C == 1) {
                __syncthreads();
                break;
            }
            // the tournament's next blocks: first <- first of CTA me - 1 (CTA 1: second of CTA 0; CTA 0 keeps
            // its own), second <- second of CTA me + 1 (the last CTA: its own first)
            cluster_barrier();
            const int nb2 = buf ^ 1;
            for (int blk = 0; blk < 2; ++blk) {
                int from, fb;
                if (blk == 0) {
                    from = me == 0 ? 0 : (int)me - 1;
                    fb = me == 1 ? 1 : 0;
                } else {
                    from = me + 1 < C ? (int)me + 1 : (int)me;
                    fb = me + 1 < C ? 1 : 0;
                }
                const uint32_t src = remote_addr(row(buf, fb, 0), from);
                uint4* dst = reinterpret_cast<uint4*>(row(nb2, blk, 0));
                const int count = b * 2 * dp / 4;
                for (int e = threadIdx.x; e < count; e += 4 * blockDim.x) {
                    uint4 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (e + u * (int)blockDim.x < count) v[u] = remote_ld16(src + 16u * (uint32_t)(e + u * blockDim.x));
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (e + u * (int)blockDim.x < count) dst[e + u * blockDim.x] = v[u];
                }
                if (threadIdx.x < kJacobiMaxWarps / 2)
                    reinterpret_cast<uint4*>(norm_s[nb2][blk])[threadIdx.x] =
                        remote_ld16(remote_addr(norm_s[buf][fb], from) + 16u * threadIdx.x);
                else if (threadIdx.x < kJacobiMaxWarps / 2 + kJacobiMaxWarps / 4)
                    reinterpret_cast<uint4*>(id_s[nb2][blk])[threadIdx.x - kJacobiMaxWarps / 2] =
                        remote_ld16(remote_addr(id_s[buf][fb], from) + 16u * (threadIdx.x - kJacobiMaxWarps / 2));
            }
            buf = nb2;
            __syncthreads();
        }
        // rotations of the sweep in every CTA (two counters, the other one cleared for the next sweep)
        int total = rotated_s[sweep & 1];
        if (C > 1) {
            total = 0;
            for (uint32_t c = 0; c < C; ++c) {
                uint32_t v;
                asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(remote_addr(&rotated_s[sweep & 1], (int)c)) : "memory");
                total += (int)v;
            }
        }
        if (total == 0) break;
        __syncthreads();
        if (threadIdx.x == 0) rotated_s[(sweep + 1) & 1] = 0;
        __syncthreads();
    }
    if (me == 0 && threadIdx.x == 0) *sweeps_out = sweep < max_sweeps ? sweep + 1 : max_sweeps + 1;
    for (int blk = 0; blk < 2; ++blk)
        for (int i = w; i < b; i += nw) {
            const int id = id_s[buf][blk][i];
            if (id < 0) continue;
            const float* src = row(buf, blk, i);
            for (int e = lane; e < d; e += 32) {
                Yh[(int64_t)id * d + e] = src[e];
                Yl[(int64_t)id * d + e] = src[dp + e];
            }
        }
    if (C > 1) cluster_barrier();                          // no CTA leaves while another may read its shared memory
}

// sigma (d, descending; zeros past the r rows) and order (the row of Y that holds each) from the
// row norms of Y; *rank_out = #{sigma_j > tau sigma_1}. One CTA of 1024 threads, bitonic sort of
// (sigma, row) pairs, ties to the lower row.
__global__ void __launch_bounds__(1024) k_sigma_rank(const double* __restrict__ Y, const int64_t* __restrict__ d_rows,
                                                     int d, double tau, double* __restrict__ sigma,
                                                     int32_t* __restrict__ order, int64_t* __restrict__ rank_out) {
    __shared__ double sv[1024];
    __shared__ int si[1024];
    __shared__ int cnt;
    const int r = (int)min(max(*d_rows, (int64_t)0), (int64_t)d);
    const int t = threadIdx.x;
    if (t == 0) cnt = 0;
    for (int i = t; i < 1024; i += blockDim.x) {
        double v = -1.0;
        if (i < r) {
            const double* y = Y + (int64_t)i * d;
            double s2 = 0.0;
            for (int j = 0; j < d; ++j) s2 = fma(y[j], y[j], s2);
            v = sqrt(s2);
        }
        sv[i] = v;
        si[i] = i;
    }
    __syncthreads();
    for (int size = 2; size <= 1024; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const int j = t ^ stride;
            if (j > t) {
                const bool desc = (t & size) == 0;
                const bool t_first = sv[t] > sv[j] || (sv[t] == sv[j] && si[t] < si[j]);
                if (t_first != desc) {
                    const double v = sv[t];
                    sv[t] = sv[j];
                    sv[j] = v;
                    const int x = si[t];
                    si[t] = si[j];
                    si[j] = x;
                }
            }
            __syncthreads();
        }
    }
    const double top = sv[0];
    if (t < d) {
        sigma[t] = t < r ? sv[t] : 0.0;
        order[t] = t < r ? si[t] : -1;
        if (t < r && top > 0.0 && sv[t] > tau * top) atomicAdd(&cnt, 1);
    }
    __syncthreads();
    if (t == 0) *rank_out = cnt;
}

// Z[:, c] = R11^{-1} b_c (k x d, row-major, ld = d): b_c = e_c for c < k, R[:k, c] for c >= k.
// One CTA per column, one thread per row, the unit-diagonal substitution of the Omega solve
// (Rs: R11's strictly upper part scaled by its diagonal and transposed).
__global__ void __launch_bounds__(1024) k_srrqr_solve(const double* __restrict__ R, const double* __restrict__ Rs,
                                                      int d, int k, double* __restrict__ Z) {
    __shared__ double xs[2];
    const int c = blockIdx.x, i = threadIdx.x;
    double x = 0.0;
    if (i < k) {
        const double b = c < k ? (i == c ? 1.0 : 0.0) : R[(int64_t)i * d + c];
        x = b / R[(int64_t)i * d + i];
    }
    const int top = c < k ? c : k - 1;               // e_c has no entries below row c
    for (int j = top; j >= 0; --j) {
        if (i == j) xs[j & 1] = x;
        __syncthreads();
        if (i < j) x = fma(-Rs[(int64_t)j * d + i], xs[j & 1], x);
    }
    if (i < k) Z[(int64_t)i * d + c] = x;
}

// wn[i] = ||e_i^T R11^{-1}||^2 (i < k); g2[j] = max(G[P_j][P_j] - ||R[:k, j]||^2, 0) (k <= j < d).
__global__ void k_srrqr_norms(const double* __restrict__ Z, const double* __restrict__ R,
                              const double* __restrict__ G, const int32_t* __restrict__ perm, int d, int k,
                              double* __restrict__ wn, double* __restrict__ g2) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < k) {
        double s = 0.0;
        for (int c = t; c < k; ++c) s = fma(Z[(int64_t)t * d + c], Z[(int64_t)t * d + c], s);
        wn[t] = s;
    } else if (t < d) {
        const int pc = perm[t];
        double s = G[(int64_t)pc * d + pc];
        for (int i = 0; i < k; ++i) s = fma(-R[(int64_t)i * d + t], R[(int64_t)i * d + t], s);
        g2[t] = s > 0.0 ? s : 0.0;
    }
}

// Largest rho^2 over i < k, k <= j < d (ties to the lower row-major index i (d - k) + (j - k)):
// per-CTA winners into part, then one CTA picks among them. out: {rho^2, i, j}.
__device__ __forceinline__ bool better(double v, long long e, double bv, long long be) {
    return v > bv || (v == bv && e < be);
}

__global__ void __launch_bounds__(256) k_srrqr_argmax(const double* __restrict__ Z, const double* __restrict__ wn,
                                                      const double* __restrict__ g2, int d, int k,
                                                      double* __restrict__ part_v, long long* __restrict__ part_e) {
    __shared__ double bv_s[256];
    __shared__ long long be_s[256];
    const long long total = (long long)k * (d - k);
    double bv = -1.0;
    long long be = total;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e / (d - k)), j = k + (int)(e % (d - k));
        const double x = Z[(int64_t)i * d + j];
        const double v = fma(x, x, g2[j] * wn[i]);
        if (better(v, e, bv, be)) {
            bv = v;
            be = e;
        }
    }
    bv_s[threadIdx.x] = bv;
    be_s[threadIdx.x] = be;
    __syncthreads();
    for (int o = blockDim.x >> 1; o > 0; o >>= 1) {
        if (threadIdx.x < o && better(bv_s[threadIdx.x + o], be_s[threadIdx.x + o], bv_s[threadIdx.x], be_s[threadIdx.x])) {
            bv_s[threadIdx.x] = bv_s[threadIdx.x + o];
            be_s[threadIdx.x] = be_s[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part_v[blockIdx.x] = bv_s[0];
        part_e[blockIdx.x] = be_s[0];
    }
}

__global__ void __launch_bounds__(256) k_srrqr_pick(const double* __restrict__ part_v, const long long* __restrict__ part_e,
                                                    int parts, int d, int k, double* __restrict__ out) {
    __shared__ double bv_s[256];
    __shared__ long long be_s[256];
    double bv = -1.0;
    long long be = 1ll << 62;
    for (int u = threadIdx.x; u < parts; u += blockDim.x)
        if (better(part_v[u], part_e[u], bv, be)) {
            bv = part_v[u];
            be = part_e[u];
        }
    bv_s[threadIdx.x] = bv;
    be_s[threadIdx.x] = be;
    __syncthreads();
    for (int o = blockDim.x >> 1; o > 0; o >>= 1) {
        if (threadIdx.x < o && better(bv_s[threadIdx.x + o], be_s[threadIdx.x + o], bv_s[threadIdx.x], be_s[threadIdx.x])) {
            bv_s[threadIdx.x] = bv_s[threadIdx.x + o];
            be_s[threadIdx.x] = be_s[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = bv_s[0];
        out[1] = (double)(be_s[0] / (d - k));
        out[2] = (double)(k + be_s[0] % (d - k));
    }
}

// perm[i] <-> perm[j] when rho^2 > phi^2 (out = {rho^2, i, j} of k_srrqr_pick).
__global__ void k_srrqr_swap(const double* __restrict__ out, double phi2, int32_t* __restrict__ perm) {
    if (threadIdx.x == 0 && out[0] > phi2) {
        const int i = (int)out[1], j = (int)out[2];
        const int32_t x = perm[i];
        perm[i] = perm[j];
        perm[j] = x;
    }
}

}  // namespace

// Y or Z (d x d), sigma, wn, g2 (d each), out (16), argmax partials (1024 values + 1024 indices),
// then 64 uint32 of barrier and rotation counts, order (d int32), the sweep count, the row versions
// of the Jacobi (d uint32, from the sweep count + 2), and the double-float rows (2 d^2 FP32).
size_t rank_scratch_doubles(int64_t d) { return (size_t)(d * d + 3 * d + 16 + 2 * 1024 + 32 + d + 8 + d + d * d + 8); }

// The cluster form: C CTAs, bmax rows a block. cudaErrorNotSupported (nothing launched) where the rows do not
// fit or no such cluster can be resident.
template <int Q>
static cudaError_t launch_jacobi_cluster(float* Yh, float* Yl, const int64_t* d_rows, int d, int C, int max_sweeps,
                                         int32_t* sweeps_out, cudaStream_t st) {
    static std::atomic<int> resident[2][64] = {};           // per (C > 8, device): 1 yes, -1 no, 0 unknown
    const int bmax = (d + 2 * C - 1) / (2 * C);
    const size_t smem = sizeof(float) * 2 * 2 * (size_t)bmax * 2 * 128 * Q;
    if (bmax > kJacobiMaxWarps || smem > 220 * 1024) return cudaErrorNotSupported;
    cudaError_t e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    std::atomic<int>* known = dev >= 0 && dev < 64 ? &resident[C > 8 ? 1 : 0][dev] : nullptr;
    if (known && known->load(std::memory_order_relaxed) < 0) return cudaErrorNotSupported;
    if ((e = cudaFuncSetAttribute(k_jacobi_cluster<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024)) != cudaSuccess)
        return e;
    if (C > 8 && cudaFuncSetAttribute(k_jacobi_cluster<Q>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return cudaErrorNotSupported;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3(32u * (unsigned)bmax);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (!known || known->load(std::memory_order_relaxed) == 0) {
        cudaLaunchConfig_t big = cfg;                        // the largest footprint of this instance
        big.blockDim = dim3(32 * kJacobiMaxWarps);
        big.dynamicSmemBytes = 220 * 1024;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, k_jacobi_cluster<Q>, &big) != cudaSuccess || clusters < 1) {
            cudaGetLastError();
            if (known) known->store(-1, std::memory_order_relaxed);
            return cudaErrorNotSupported;
        }
        if (known) known->store(1, std::memory_order_relaxed);
    }
    e = cudaLaunchKernelEx(&cfg, k_jacobi_cluster<Q>, Yh, Yl, d_rows, d, bmax, max_sweeps, sweeps_out);
    return e;
}

cudaError_t launch_svd_rank(const double* R, const int64_t* d_rows, int64_t d, double tau, double* Y, float* Yhl,
                            unsigned* work, double* sigma, int32_t* order, int64_t* rank_out, int32_t* sweeps_out,
                            unsigned* version, int32_t* status, int num_sms, cudaStream_t st) {
    cudaError_t e;
    constexpr int kMaxSweeps = 40;
    if (d > 1024) return cudaErrorInvalidValue;
    float* Yh = Yhl;
    float* Yl = Yhl + d * d;
    int cg = (int)((d * d + 255) / 256);
    if (cg > 152 * 8) cg = 152 * 8;
    k_split_rows<<<cg, 256, 0, st>>>(R, d * d, Yh, Yl);
    // one cluster of 1 to 16 CTAs (blocks of at least 8 rows) where its shared memory holds the rows twice
    const int C = d <= 16 ? 1 : d <= 32 ? 2 : d <= 64 ? 4 : d <= 128 ? 8 : 16;
    e = d <= 128 ? launch_jacobi_cluster<1>(Yh, Yl, d_rows, (int)d, C, kMaxSweeps, sweeps_out, st)
      : d <= 256 ? launch_jacobi_cluster<2>(Yh, Yl, d_rows, (int)d, C, kMaxSweeps, sweeps_out, st)
      : d <= 384 ? launch_jacobi_cluster<3>(Yh, Yl, d_rows, (int)d, C, kMaxSweeps, sweeps_out, st)
                 : cudaErrorNotSupported;
    if (e != cudaSuccess && e != cudaErrorNotSupported) return e;
    if (e == cudaErrorNotSupported) {
        unsigned* barrier = work;
        unsigned* rotated = work + 1;
        if ((e = cudaMemsetAsync(work, 0, sizeof(unsigned) * (1 + kMaxSweeps), st)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(version, 0, sizeof(unsigned) * (size_t)d, st)) != cudaSuccess) return e;
        int di = (int)d, ms = kMaxSweeps;
        void* kargs[] = {&Yh, &Yl, (void*)&d_rows, &di, &ms, &rotated, &barrier, &version, &status, &sweeps_out};
        const void* fn = d <= 256 ? (const void*)k_jacobi_rows<1>
                       : d <= 512 ? (const void*)k_jacobi_rows<2> : (const void*)k_jacobi_rows<4>;
        int occ = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, 256, 0)) != cudaSuccess) return e;
        int grid = (int)((d + 1) / 2);                      // one CTA a pair where they fit
        const int cap = num_sms * (occ < 1 ? 1 : occ);
        if (grid > cap) grid = cap;
        if (grid < 1) grid = 1;
        if ((e = cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(256), kargs, 0, st)) != cudaSuccess) return e;
    }
    k_join_rows<<<cg, 256, 0, st>>>(Yh, Yl, d * d, Y);
    k_sigma_rank<<<1, 1024, 0, st>>>(Y, d_rows, (int)d, tau, sigma, order, rank_out);
    return cudaGetLastError();
}

cudaError_t launch_srrqr_step(const double* R, const double* Rs, const double* G, int32_t* perm, int64_t d, int64_t k,
                              double phi, double* Z, double* wn, double* g2, double* part_v, long long* part_e,
                              double* out, cudaStream_t st) {
    if (k < 1 || k >= d || d > 1024) return cudaErrorInvalidValue;
    k_srrqr_solve<<<(unsigned)d, (unsigned)((k + 31) / 32 * 32), 0, st>>>(R, Rs, (int)d, (int)k, Z);
    k_srrqr_norms<<<(unsigned)((d + 255) / 256), 256, 0, st>>>(Z, R, G, perm, (int)d, (int)k, wn, g2);
    const long long total = k * (d - k);
    int parts = (int)((total + 255) / 256);
    if (parts > 1024) parts = 1024;
    k_srrqr_argmax<<<(unsigned)parts, 256, 0, st>>>(Z, wn, g2, (int)d, (int)k, part_v, part_e);
    k_srrqr_pick<<<1, 256, 0, st>>>(part_v, part_e, parts, (int)d, (int)k, out);
    k_srrqr_swap<<<1, 32, 0, st>>>(out, phi * phi, perm);
    return cudaGetLastError();
}

}  // namespace lev
