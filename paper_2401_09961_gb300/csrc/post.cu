// Post-processing of an unwrapped image (Sec. 4.5): the "rounded IRLS" output, 2pi-congruent to
// the input, and the best-shift error against a reference unwrapping.  The reductions are
// deterministic last-block sums to FP64 accuracy; the per-pixel integer decisions are float32, one
// correctly rounded operation at a time.
//
// FP64 arithmetic runs at a 64th of the float32 rate on this part, so the per-pixel work of the
// reductions is float32 with error-free transformations (pairs hi + lo), and FP64 enters once per
// several pixels.
#include <algorithm>
#include <initializer_list>

#include "irls_internal.cuh"
#include "reduce.cuh"

namespace irls {

namespace {

constexpr int kPostThreads = 256;
constexpr float kTwoPiF = 6.28318530717958647692f;   // 2pi rounded to float32

// Four consecutive values (fewer at the end of the array: zeros); vec: 16-byte aligned.
__device__ __forceinline__ void load4(const float* __restrict__ p, size_t i, int m, bool vec,
                                      float (&x)[4]) {
    if (vec && m == 4) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p + i));
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = q < m ? __ldg(p + i + q) : 0.f;
    }
}
template <class T, class T4>
__device__ __forceinline__ void store4(T* __restrict__ p, size_t i, int m, bool vec,
                                       const T (&x)[4]) {
    if (vec && m == 4) {
        T4 v;
        v.x = x[0]; v.y = x[1]; v.z = x[2]; v.w = x[3];
        *reinterpret_cast<T4*>(p + i) = v;
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q < m) p[i + q] = x[q];
    }
}

// ---- circular mean offset -------------------------------------------------------------------
// cos and sin of the N-th parts of the circle, each split into four floats of which the first
// three are multiples of 2^-12, 2^-24 and 2^-36 (at most 13 bits each), so that float32 sums of up
// to kCircRun of them are exact, and whose total is within 2^-61 of the value.
constexpr int kCircN = 2048, kCircRun = 1024;
struct CircEntry {
    float c[4], s[4];
};

__device__ __forceinline__ void split_circ(double v, float (&o)[4]) {
    double step = 4096.0;
#pragma unroll
    for (int q = 0; q < 3; ++q, step *= 4096.0) {
        o[q] = (float)(rint(v * step) / step);
        v -= (double)o[q];
    }
    o[3] = (float)v;
}

__global__ void k_build_circle(CircEntry* t) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kCircN) return;
    double s, c;
    sincospi(2.0 * (double)k / (double)kCircN, &s, &c);
    split_circ(c, t[k].c);
    split_circ(s, t[k].s);
}

// d = k P + delta with P = 2 pi / kCircN and |delta| at most half a part (or a rounding more), as delta = hi + lo: every
// difference is error-free (two-sums, products with their FMA remainder), lo within a few 1e-18.
// P as three floats; |d| below 8192 keeps k an exact float.
__device__ __forceinline__ void reduce_circ(float dh, float dl, int& k, float& hi, float& lo) {
    const float kP1 = 0x1.921fb6p-9f, kP2 = -0x1.777a5cp-34f, kP3 = -0x1.ee59dap-59f;
    const float n = rintf(__fmul_rn(dh, 0x1.45f306p+8f));
    k = (int)n;
    float p, pe, q, qe, s, t0, t1, t2, t3;
    two_prod(n, kP1, p, pe);
    two_prod(n, kP2, q, qe);
    two_sum(dh, -p, s, t0);
    two_sum(s, -pe, s, t1);
    two_sum(s, dl, s, t2);
    two_sum(s, -q, s, t3);
    const float r = __fadd_rn(__fadd_rn(t0, t1),
                              __fadd_rn(__fadd_rn(t2, t3), __fmaf_rn(-n, kP3, -qe)));
    two_sum(s, r, hi, lo);
}

// sum cos(U - X), sum sin(U - X); the last block stores the circular mean offset c = atan2(S, C)
// in st->aux[0].  cos(a + delta) = C + (C (cos delta - 1) - S sin delta) with a table entry
// (C, S) and |delta| < 0.0016: the entries are summed exactly, the small correction as a
// compensated float32 pair; both go to FP64 every kCircRun pixels of a thread.  The sums are
// within FP64 rounding of the exact ones.  About 110 float32 operations a pixel bound it: 4096^2
// in 0.1 ms, where FP64 sincos took 1.1 ms.  Differences of 8192 rad and more, and values that
// are not finite, take FP64 sincos.
constexpr int kCircThreads = 512;
__global__ void __launch_bounds__(kCircThreads, 2)
k_circ_offset(const float* __restrict__ U, const float* __restrict__ X, size_t n, int vec,
              const CircEntry* __restrict__ table, DevState* st, double* partials) {
    extern __shared__ __align__(16) float4 tab[];   // [2 k]: c, [2 k + 1]: s
    for (int e = threadIdx.x; e < 2 * kCircN; e += kCircThreads)
        tab[e] = __ldg(reinterpret_cast<const float4*>(table) + e);
    __syncthreads();
    double c = 0.0, s = 0.0;
    float ct[4] = {0, 0, 0, 0}, sn[4] = {0, 0, 0, 0};   // table sums
    CSum cc, ss;                                        // corrections
    float cl = 0.f, sl = 0.f;                           // their low parts
    int run = 0;
    const size_t quads = (n + 3) / 4;
    for (size_t t = blockIdx.x * (size_t)kCircThreads + threadIdx.x; t < quads;
         t += (size_t)gridDim.x * kCircThreads) {
        const size_t i = 4 * t;
        const int m = n - i < 4 ? (int)(n - i) : 4;
        float u[4], x[4];
        load4(U, i, m, vec, u);
        load4(X, i, m, vec, x);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (e >= m) break;
            float dh, dl;
            two_sum(u[e], -x[e], dh, dl);
            if (!(fabsf(dh) < 8192.f)) {
                double a, b;
                sincos((double)u[e] - (double)x[e], &a, &b);
                c += b;
                s += a;
                continue;
            }
            int k;
            float h, l;
            reduce_circ(dh, dl, k, h, l);
            const float4 C = tab[2 * (k & (kCircN - 1))], S = tab[2 * (k & (kCircN - 1)) + 1];
            ct[0] += C.x; ct[1] += C.y; ct[2] += C.z; ct[3] += C.w;
            sn[0] += S.x; sn[1] += S.y; sn[2] += S.z; sn[3] += S.w;
            // 1 - cos delta and sin delta as pairs
            float h2, l2;
            two_prod(h, h, h2, l2);
            l2 = __fmaf_rn(2.f * h, l, l2);
            const float mh = -0.5f * h2;
            const float ml = __fmaf_rn(h2 * h2, __fmaf_rn(h2, -1.f / 720.f, 1.f / 24.f), -0.5f * l2);
            const float sl3 = __fmaf_rn(h * h2, __fmaf_rn(h2, 1.f / 120.f, -1.f / 6.f), l);
            // the entry as a pair: the first two parts add exactly
            const float ch = C.x + C.y, c2 = C.z + C.w, sh = S.x + S.y, s2 = S.z + S.w;
            float a, ae, b, be, q, t0;
            two_prod(ch, mh, a, ae);
            two_prod(sh, h, b, be);
            two_sum(a, -b, q, t0);
            cc.add(q);
            cl += t0 + ((ae - be) + (__fmaf_rn(ch, ml, c2 * mh) - __fmaf_rn(sh, sl3, s2 * h)));
            two_prod(sh, mh, a, ae);
            two_prod(ch, h, b, be);
            two_sum(a, b, q, t0);
            ss.add(q);
            sl += t0 + ((ae + be) + (__fmaf_rn(sh, ml, s2 * mh) + __fmaf_rn(ch, sl3, c2 * h)));
        }
        if ((run += 4) == kCircRun || t + (size_t)gridDim.x * kCircThreads >= quads) {
            c += (((double)ct[3] + ct[2]) + ct[1]) + ct[0] + (cc.value() + cl);
            s += (((double)sn[3] + sn[2]) + sn[1]) + sn[0] + (ss.value() + sl);
#pragma unroll
            for (int q = 0; q < 4; ++q) ct[q] = sn[q] = 0.f;
            cc = ss = CSum();
            cl = sl = 0.f;
            run = 0;
        }
    }
    double v[2] = {c, s}, tot[2];
    if (grid_reduce<2>(v, partials, &st->counter, tot, gridDim.x, blockIdx.x) && threadIdx.x == 0)
        st->aux[0] = atan2(tot[1], tot[0]);
}

// K = rint(((U - c) - X) / 2pi), U_round = X + 2pi K
__global__ void __launch_bounds__(kPostThreads)
k_round_congruent(const float* __restrict__ U, const float* __restrict__ X, size_t n, int vec,
                  const DevState* st, float* __restrict__ Ur, int* __restrict__ K) {
    const float c = (float)st->aux[0];
    const size_t quads = (n + 3) / 4;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < quads;
         t += (size_t)gridDim.x * blockDim.x) {
        const size_t i = 4 * t;
        const int m = n - i < 4 ? (int)(n - i) : 4;
        float u[4], x[4], r[4];
        int kk[4];
        load4(U, i, m, vec, u);
        load4(X, i, m, vec, x);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float d = __fsub_rn(__fsub_rn(u[e], c), x[e]);
            const float k = rintf(__fdiv_rn(d, kTwoPiF));
            r[e] = __fadd_rn(x[e], __fmul_rn(kTwoPiF, k));
            kk[e] = (int)k;
        }
        if (Ur) store4<float, float4>(Ur, i, m, vec, r);
        if (K) store4<int, int4>(K, i, m, vec, kk);
    }
}

// alpha = mean(Xu - U) (FP64) into st->aux[1]: four differences and their rounding remainders as
// one pair, then FP64.  Four pixels with a difference that is not finite, or whose sum could
// overflow, go to FP64 one by one.
__global__ void __launch_bounds__(kPostThreads)
k_shift_mean(const float* __restrict__ U, const float* __restrict__ Xu, size_t n, int vec,
             DevState* st, double* partials) {
    double s = 0.0;
    const size_t quads = (n + 3) / 4;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < quads;
         t += (size_t)gridDim.x * blockDim.x) {
        const size_t i = 4 * t;
        const int m = n - i < 4 ? (int)(n - i) : 4;
        float u[4], x[4], d[4], l[4];
        load4(U, i, m, vec, u);
        load4(Xu, i, m, vec, x);
        bool in_range = true;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            two_sum(x[e], -u[e], d[e], l[e]);
            in_range &= fabsf(d[e]) < 0x1p120f;
        }
        if (!in_range) {
            for (int e = 0; e < m; ++e) s += (double)x[e] - (double)u[e];
            continue;
        }
        float a, b, h, e0, e1, e2;
        two_sum(d[0], d[1], a, e0);
        two_sum(d[2], d[3], b, e1);
        two_sum(a, b, h, e2);
        s += (double)h + (double)(((l[0] + l[1]) + (l[2] + l[3])) + ((e0 + e1) + e2));
    }
    double v[1] = {s}, tot[1];
    if (grid_reduce<1>(v, partials, &st->counter, tot, gridDim.x, blockIdx.x) && threadIdx.x == 0)
        st->aux[1] = tot[0] / (double)n;
}

// E = (Xu - U) - alpha (float32), sum of ((Xu - U) - alpha)^2 into st->aux[2].  The error of a pixel
// is the exact difference (a pair) less alpha (three floats), every step error-free and the pair
// that remains normalised: alpha may be far larger than the errors (images of different offsets),
// and the second part is squared with the first.  Squares are pairs, FP64 every four pixels.  Four
// pixels whose largest error is not finite or whose squares could overflow, or lose their
// remainders below the smallest floats, go to FP64 one by one.  (Without the third float, the second
// normalisation and the range check the two calls at 4096^2 take 283 us instead of 292, but an offset
// of 1000 rad over 1e-3 rad of noise puts rms off by 2e-4.)
__global__ void __launch_bounds__(kPostThreads)
k_shift_error(const float* __restrict__ U, const float* __restrict__ Xu, size_t n, int vec,
              DevState* st, double* partials, float* __restrict__ E) {
    const double alpha = st->aux[1];
    const float a1 = (float)alpha, a2 = (float)(alpha - (double)a1);
    const float a3 = (float)((alpha - (double)a1) - (double)a2);
    double s2 = 0.0;
    const size_t quads = (n + 3) / 4;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < quads;
         t += (size_t)gridDim.x * blockDim.x) {
        const size_t i = 4 * t;
        const int m = n - i < 4 ? (int)(n - i) : 4;
        float u[4], x[4], o[4], q[4], r[4];
        load4(U, i, m, vec, u);
        load4(Xu, i, m, vec, x);
        float most = 0.f;
        bool in_range = true;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float d, l, p, w, c0, c1, c2, c3, hi, lo;
            two_sum(x[e], -u[e], d, l);
            o[e] = __fsub_rn(d, a1);
            two_sum(d, -a1, p, c0);
            two_sum(l, -a2, c1, c2);
            two_sum(c0, c1, w, c3);
            two_sum(p, w, hi, lo);
            two_sum(hi, __fadd_rn(lo, __fsub_rn(__fadd_rn(c2, c3), a3)), p, w);
            two_prod(p, p, q[e], r[e]);
            r[e] = __fmaf_rn(2.f * p, w, __fmaf_rn(w, w, r[e]));
            if (e < m) {
                in_range &= fabsf(p) < 0x1p60f;
                most = fmaxf(most, fabsf(p));
            } else {
                q[e] = r[e] = 0.f;
            }
        }
        if (E) store4<float, float4>(E, i, m, vec, o);
        if (!in_range || (most < 0x1p-45f && most != 0.f)) {
            for (int e = 0; e < m; ++e) {
                const double f = ((double)x[e] - (double)u[e]) - alpha;
                s2 += f * f;
            }
            continue;
        }
        float a, b, h, e0, e1, e2;
        two_sum(q[0], q[1], a, e0);
        two_sum(q[2], q[3], b, e1);
        two_sum(a, b, h, e2);
        s2 += (double)h + (double)(((r[0] + r[1]) + (r[2] + r[3])) + ((e0 + e1) + e2));
    }
    double v[1] = {s2}, tot[1];
    if (grid_reduce<1>(v, partials, &st->counter, tot, gridDim.x, blockIdx.x) && threadIdx.x == 0)
        st->aux[2] = tot[0];
}

int post_blocks(size_t n, int max_blocks, int threads, int most) {
    const size_t b = (n + 4 * (size_t)threads - 1) / (4 * (size_t)threads);
    return (int)std::max<size_t>(1, std::min({b, (size_t)most, (size_t)max_blocks}));
}

int all_aligned16(std::initializer_list<const void*> ps) {
    for (const void* p : ps)
        if (reinterpret_cast<uintptr_t>(p) & 15) return 0;
    return 1;
}

}  // namespace

size_t circle_bytes() { return kCircN * sizeof(CircEntry); }

cudaError_t build_circle(void* mem) {
    k_build_circle<<<kCircN / 256, 256>>>(static_cast<CircEntry*>(mem));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_circ_offset, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)circle_bytes());
}

cudaError_t launch_round_congruent(const float* U, const float* X, size_t n, const void* circle,
                                   DevState* st, double* partials, int max_blocks, float* Ur,
                                   int* K, cudaStream_t s) {
    const int nc = post_blocks(n, max_blocks, kCircThreads, 304);   // two blocks an SM
    k_circ_offset<<<nc, kCircThreads, circle_bytes(), s>>>(
        U, X, n, all_aligned16({U, X}), static_cast<const CircEntry*>(circle), st, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_round_congruent<<<post_blocks(n, 1 << 30, kPostThreads, 4096), kPostThreads, 0, s>>>(
        U, X, n, all_aligned16({U, X, Ur, K}), st, Ur, K);
    return cudaGetLastError();
}

cudaError_t launch_best_shift(const float* U, const float* Xu, size_t n, DevState* st,
                              double* partials, int max_blocks, float* E, cudaStream_t s) {
    const int nb = post_blocks(n, max_blocks, kPostThreads, 1216);   // eight blocks an SM
    k_shift_mean<<<nb, kPostThreads, 0, s>>>(U, Xu, n, all_aligned16({U, Xu}), st, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_shift_error<<<nb, kPostThreads, 0, s>>>(U, Xu, n, all_aligned16({U, Xu, E}), st, partials, E);
    return cudaGetLastError();
}

}  // namespace irls
