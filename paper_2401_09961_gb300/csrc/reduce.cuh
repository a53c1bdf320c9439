// Deterministic grid-wide FP64 reductions finished by the last block of a launch.
#pragma once

#include <cuda_runtime.h>

namespace irls {

// Compensated float32 sum (Knuth's two-sum): hi + lo carries the running sum of the added terms
// with an error that does not grow with their number, at seven float32 operations per added
// term.  The per-thread partials of every inner product of the CG iteration are accumulated in
// one (each added term is a single value or a partial of at most four values of one image row),
// then carried into the FP64 warp, block and grid sums as (double)hi + (double)lo.  The
// intrinsics keep the compiler from contracting or reordering the error terms.
struct CSum {
    float hi, lo;
    __device__ __forceinline__ CSum() : hi(0.f), lo(0.f) {}
    __device__ __forceinline__ void add(float x) {
        const float s = __fadd_rn(hi, x);
        const float bp = __fsub_rn(s, hi);
        const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
        hi = s;
        lo = __fadd_rn(lo, e);
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// Error-free transformations in float32: a + b = s + e and a * b = p + e exactly (Knuth's
// two-sum; the product's error from one fused multiply-add).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}

// The terms of A x that cancel (Sec. 3.2, the vectorised A), carried as hi + lo pairs so that
// the difference keeps the accuracy of its float32 operands:
//   s * (y0 + y1 + y2 + y3)        (the U row: s = 1/tau times a sum of four edge terms)
//   d * v - s * y                   (a V row: D V minus the penalty term)
__device__ __forceinline__ void sum4_scaled(float s, float y0, float y1, float y2, float y3,
                                            float& hi, float& lo) {
    float t, e1, e2, e3;
    two_sum(y0, y1, t, e1);
    two_sum(t, y2, t, e2);
    two_sum(t, y3, t, e3);
    two_prod(s, t, hi, lo);
    lo = __fmaf_rn(s, __fadd_rn(__fadd_rn(e1, e2), e3), lo);
}
__device__ __forceinline__ void diff_prod(float d, float v, float s, float y, float& hi,
                                          float& lo) {
    float p1, e1, p2, e2, e3;
    two_prod(d, v, p1, e1);
    two_prod(s, y, p2, e2);
    two_sum(p1, -p2, hi, e3);
    lo = __fadd_rn(e3, __fsub_rn(e1, e2));
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sums of NV per-lane values over a warp: lane k < NV returns the k-th sum.  The values are halved
// between partner lanes at each of the first levels (each lane keeps the half its lane bit
// names), so that NV = 5 takes 4 + 2 + 1 + 1 + 1 FP64 additions a lane instead of 25: the FP64
// pipe (two additions a cycle and SM) is what the block ends of the small launches wait for.
template <int NV>
__device__ __forceinline__ double warp_sums(const double (&v)[NV]) {
    constexpr int P = NV <= 1 ? 1 : NV <= 2 ? 2 : NV <= 4 ? 4 : 8;
    double x[P];
#pragma unroll
    for (int k = 0; k < P; ++k) x[k] = k < NV ? v[k < NV ? k : 0] : 0.0;
    const int lane = threadIdx.x & 31;
    int o = 1;
#pragma unroll
    for (int n = P / 2; n >= 1; n /= 2, o *= 2) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            // keep the values whose index bit (from the top of P) equals the lane's bit
            const double keep = up ? x[k + n] : x[k], give = up ? x[k] : x[k + n];
            x[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    double t = x[0];
#pragma unroll
    for (; o < 32; o *= 2) t += __shfl_xor_sync(0xffffffffu, t, o);
    // lane bits (1, 2, 4) chose the value's index bits from the top: undo the reversal
    int src = 0;
#pragma unroll
    for (int b = 1, n = P / 2; n >= 1; b *= 2, n /= 2) src |= (lane & n) ? b : 0;
    return P == 1 ? t : __shfl_sync(0xffffffffu, t, src);
}

// Block coordinates of one problem's launch grid: the launch's own grid for a single image, or
// the problem's share of a batched launch (several images in one grid).
struct Blk {
    int bx, by;
    unsigned nblk, bid;
};

__device__ __forceinline__ Blk single_blk() {
    Blk b;
    b.bx = blockIdx.x;
    b.by = blockIdx.y;
    b.nblk = gridDim.x * gridDim.y;
    b.bid = blockIdx.x + gridDim.x * blockIdx.y;
    return b;
}

// Sums NV per-thread values over the problem's blocks (nblk of them, this one is bid).  Every
// block writes its partial to partials[k * nblk + bid]; the block that takes the last ticket
// adds the partials in a fixed order (so a re-run is bit-identical) and returns true with `tot`
// valid in its first thread.  Other blocks return false.  The ticket counter is reset by the last block, so the
// next launch on the same stream can reuse it.  There is no waiting: a block that is not last
// simply leaves.
//
// With UNITS the block holds several consecutive units of the image's rows, each with a partial
// of its own: unit_done puts a warp's sums of one unit into shared memory, and the block writes
// its units' partials at unit * gx + bx, so that the sum does not depend on how many units a
// block holds.
constexpr int kMaxUnits = 32;   // units a block can hold (rows per block of a batch at most 32)

template <int NV>
struct UnitSums {
    double w[kMaxUnits][NV][4];   // four warps
};
template <>
struct UnitSums<0> {};            // a block of one unit

template <int NV>
__device__ __forceinline__ void unit_done(UnitSums<NV>& s, int unit, const double (&v)[NV]) {
    const int lane = threadIdx.x & 31;
    const double t = warp_sums<NV>(v);
    if (lane < NV) s.w[unit][lane][threadIdx.x >> 5] = t;
}

// The last block's sum of n partials per value; tot valid in its first thread.
template <int NV>
__device__ __forceinline__ void sum_partials(double (&sw)[NV][32], const double* partials,
                                             double (&tot)[NV], unsigned n) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nthr = blockDim.x * blockDim.y;
    const int lane = tid & 31, warp = tid >> 5, nwarp = (nthr + 31) >> 5;
    double s[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) s[k] = 0.0;
    for (unsigned b = tid; b < n; b += nthr) {
#pragma unroll
        for (int k = 0; k < NV; ++k) s[k] += __ldcg(&partials[(size_t)k * n + b]);
    }
    const double t = warp_sums<NV>(s);
    if (lane < NV) sw[lane][warp] = t;
    __syncthreads();
    if (tid != 0) return;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double x = 0.0;
        for (int w = 0; w < nwarp; ++w) x += sw[k][w];
        tot[k] = x;
    }
}

template <int NV>
__device__ bool grid_reduce(const double (&v)[NV], double* partials, unsigned int* counter,
                            double (&tot)[NV], unsigned nblk, unsigned bid) {
    __shared__ double sw[NV][32];
    __shared__ int s_last;
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nthr = blockDim.x * blockDim.y;
    const int lane = tid & 31, warp = tid >> 5, nwarp = (nthr + 31) >> 5;
    const double t = warp_sums<NV>(v);
    if (lane < NV) sw[lane][warp] = t;
    __syncthreads();
    if (tid < NV) {
        double s = 0.0;
        for (int w = 0; w < nwarp; ++w) s += sw[tid][w];
        __stcg(&partials[(size_t)tid * nblk + bid], s);
    }
    if (warp == 0) {
        __threadfence();
        __syncwarp();
        if (lane == 0) s_last = atomicAdd(counter, 1u) == nblk - 1u;
    }
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
    sum_partials<NV>(sw, partials, tot, nblk);
    if (tid == 0) *counter = 0u;
    return true;
}

// grid_reduce over units: the block's units are u0 .. u0 + nu - 1 (their warps' sums in `s`) of
// the image's n_units row units, in column bx of gx; 128 threads.
template <int NV>
__device__ bool grid_reduce_units(const UnitSums<NV>& s, double* partials, unsigned int* counter,
                                  double (&tot)[NV], const Blk& blk, int gx, int u0, int nu,
                                  int n_units) {
    __shared__ double sw[NV][32];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned n = (unsigned)(gx * n_units);
    __syncthreads();
    for (int e = tid; e < nu * NV; e += blockDim.x) {
        const int u = e / NV, k = e % NV;
        const double* w = s.w[u][k];
        __stcg(&partials[(size_t)k * n + (size_t)(u0 + u) * gx + blk.bx],
               ((w[0] + w[1]) + w[2]) + w[3]);
    }
    __threadfence();
    __syncthreads();
    if (warp == 0 && lane == 0) {
        __threadfence();
        s_last = atomicAdd(counter, 1u) == blk.nblk - 1u;
    }
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
    sum_partials<NV>(sw, partials, tot, n);
    if (tid == 0) *counter = 0u;
    return true;
}

}  // namespace irls
