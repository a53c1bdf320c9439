// Laplacian-block preconditioner of Sec. 3.3 by fast transforms: the same map as the dense
// products, z_U = P_N [ (P_N^T (tau r_U) P_M) / (l_i + m_j) ] P_M^T with the (0,0) entry set to
// zero, with every orthonormal DCT-II (P^T x) and DCT-III (P y) evaluated through a complex FFT
// of the same length (Makhoul's even/odd reordering) in float32 on the CUDA cores.
//
// Three launches per application, each one pass over a float32 plane:
//   rows_fwd  T[i][l]   = tau * DCT-II along the row i of r_U
//   cols      T[.][l]   = DCT-III( DCT-II(T[.][l]) / (l_k + m_l) ) per column l, in place;
//             rho_U     = sum_kl S_kl^2 / (tau (l_k + m_l)) = r_U^T z_U (Parseval), folded into
//                         the CG scalars by the last block
//   rows_inv  z_U[i][.] = DCT-III along the row i of T
// Two real sequences share one complex transform (the first as the real part, the second as the
// imaginary part); their spectra separate by the conjugate symmetry of a real sequence's DFT.
// The complex FFT is a Stockham auto-sort in shared memory; a thread holds a butterfly's values in
// registers between a stage's two barriers.  Lengths to 8192 run two transforms a thread (four
// rows or columns, "quads" below); rows of 16000 and 16384 elements, whose quads would not fit
// shared memory, one.  Lengths: powers of two, and 2000, 4000, 8000, 16000.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "irls_internal.cuh"
#include "reduce.cuh"

namespace irls {

namespace {

constexpr int kFftMinN = 64;
constexpr int kFftMaxRowN = 16384;   // row transforms
constexpr int kFftMaxColN = 8192;    // column transforms

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "sub.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

// ---- in-register DFTs (forward sign: X_q = sum_r v_r exp(-2 pi i r q / R)) --------------------
template <int R>
__device__ __forceinline__ void dft(float2* v);

template <>
__device__ __forceinline__ void dft<4>(float2* v) {
    const float2 s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
    const float2 s13 = cadd(v[1], v[3]), d13 = csub(v[1], v[3]);
    v[0] = cadd(s02, s13);
    v[2] = csub(s02, s13);
    v[1] = make_float2(d02.x + d13.y, d02.y - d13.x);   // d02 - i d13
    v[3] = make_float2(d02.x - d13.y, d02.y + d13.x);   // d02 + i d13
}

constexpr float kR2 = 0.70710678118654752f;    // cos(pi/4)
constexpr float kC8 = 0.92387953251128674f;    // cos(pi/8)
constexpr float kS8 = 0.38268343236508977f;    // sin(pi/8)

template <>
__device__ __forceinline__ void dft<8>(float2* v) {
    float2 e[4] = {v[0], v[2], v[4], v[6]};
    float2 o[4] = {v[1], v[3], v[5], v[7]};
    dft<4>(e);
    dft<4>(o);
    o[1] = make_float2((o[1].x + o[1].y) * kR2, (o[1].y - o[1].x) * kR2);   // * exp(-i pi/4)
    o[2] = make_float2(o[2].y, -o[2].x);                                    // * -i
    o[3] = make_float2((o[3].y - o[3].x) * kR2, -(o[3].x + o[3].y) * kR2);  // * exp(-3 i pi/4)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = cadd(e[k], o[k]);
        v[k + 4] = csub(e[k], o[k]);
    }
}

// Length 16 as 4 x 4: DFT4 over n2 of v[n1 + 4 n2] for each n1, twiddle exp(-2 pi i n1 k2 / 16),
// DFT4 over n1; output k2 + 4 k1.
template <>
__device__ __forceinline__ void dft<16>(float2* v) {
    float2 y[4][4];
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) {
        float2 c[4] = {v[n1], v[n1 + 4], v[n1 + 8], v[n1 + 12]};
        dft<4>(c);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) y[n1][k2] = c[k2];
    }
    // exp(-2 pi i e / 16) for e = n1 k2 in {1, 2, 3, 4, 6, 9}
    y[1][1] = cmul(y[1][1], make_float2(kC8, -kS8));
    y[1][2] = cmul(y[1][2], make_float2(kR2, -kR2));
    y[1][3] = cmul(y[1][3], make_float2(kS8, -kC8));
    y[2][1] = cmul(y[2][1], make_float2(kR2, -kR2));
    y[2][2] = make_float2(y[2][2].y, -y[2][2].x);
    y[2][3] = cmul(y[2][3], make_float2(-kR2, -kR2));
    y[3][1] = cmul(y[3][1], make_float2(kS8, -kC8));
    y[3][2] = cmul(y[3][2], make_float2(-kR2, -kR2));
    y[3][3] = cmul(y[3][3], make_float2(-kC8, kS8));
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) {
        float2 c[4] = {y[0][k2], y[1][k2], y[2][k2], y[3][k2]};
        dft<4>(c);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) v[k2 + 4 * k1] = c[k1];
    }
}

// Length 5: X_0 = v_0 + t1 + t2, X_{1,4} = a1 -/+ i b1, X_{2,3} = a2 -/+ i b2 with
// t1 = v1 + v4, t2 = v2 + v3, a1 = v0 + c1 t1 + c2 t2, a2 = v0 + c2 t1 + c1 t2,
// b1 = s1 (v1 - v4) + s2 (v2 - v3), b2 = s2 (v1 - v4) - s1 (v2 - v3), c_k + i s_k = exp(2 pi i k / 5).
constexpr float kC51 = 0.30901699437494745f, kC52 = -0.80901699437494734f;
constexpr float kS51 = 0.95105651629515353f, kS52 = 0.58778525229247325f;
template <>
__device__ __forceinline__ void dft<5>(float2* v) {
    const float2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    const float2 t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
    const float2 a1 = make_float2(v[0].x + kC51 * t1.x + kC52 * t2.x, v[0].y + kC51 * t1.y + kC52 * t2.y);
    const float2 a2 = make_float2(v[0].x + kC52 * t1.x + kC51 * t2.x, v[0].y + kC52 * t1.y + kC51 * t2.y);
    const float2 b1 = make_float2(kS51 * t3.x + kS52 * t4.x, kS51 * t3.y + kS52 * t4.y);
    const float2 b2 = make_float2(kS52 * t3.x - kS51 * t4.x, kS52 * t3.y - kS51 * t4.y);
    v[0] = cadd(v[0], cadd(t1, t2));
    v[1] = make_float2(a1.x + b1.y, a1.y - b1.x);   // a1 - i b1
    v[4] = make_float2(a1.x - b1.y, a1.y + b1.x);   // a1 + i b1
    v[2] = make_float2(a2.x + b2.y, a2.y - b2.x);
    v[3] = make_float2(a2.x - b2.y, a2.y + b2.x);
}

// ---- shared-memory layouts of NF complex sequences of length N ------------------------------
// Pair: element m of transform f as one float2 (row 2f, row 2f + 1), one float2 of padding
// every 16 (the stages' strided accesses and the reordered stores of the load fall on distinct
// banks).  Row transforms.
template <int N, int NF>
struct PairL {
    static constexpr int P2 = N + N / 16;
    static constexpr int FLOATS = NF * 2 * P2;
    __device__ static __forceinline__ int off(int f, int m) { return 2 * (f * P2 + m + (m >> 4)); }
    __device__ static __forceinline__ float2 ld(const float* s, int f, int m) {
        return *reinterpret_cast<const float2*>(s + off(f, m));
    }
    __device__ static __forceinline__ void st(float* s, int f, int m, float2 v) {
        *reinterpret_cast<float2*>(s + off(f, m)) = v;
    }
};
// Where x_i goes in the even/odd reordered sequence v of a length-N DCT: v_m = x_{2m} (m < N/2),
// x_{2N-1-2m} (m >= N/2).
template <int N>
__device__ __forceinline__ int reorder_pos(int i) { return (i & 1) ? N - 1 - (i >> 1) : (i >> 1); }

// exp(-2 pi i e / N) from the two-level table in shared memory: lo[e % 64] * hi[e / 64].
template <int N>
__device__ __forceinline__ float2 twiddle(const float2* tws, int e) {
    return cmul(tws[e & 63], tws[64 + (e >> 6)]);
}

// Entries of the two-level twiddle table of length N: 64 low and ceil(N / 64) high.
template <int N>
struct TwN {
    static constexpr int V = 64 + (N + 63) / 64;
    static constexpr int PADDED = (V + 1) & ~1;   // a 16-byte multiple
};

// Copies the two-level twiddle table of length N into shared memory.
template <int N, int T>
__device__ __forceinline__ void load_twiddles(float2* tws, const float2* __restrict__ tw) {
    for (int e = threadIdx.x; e < TwN<N>::V; e += T)
        tws[e] = e < 64 ? __ldg(&tw[e]) : __ldg(&tw[(e - 64) * 64]);
}

// Stockham stages of NF forward complex FFTs of length N in shared memory (layout L), from the
// stage whose sub-transforms have length NS; tws is the two-level table of exp(-2 pi i m / N).
// Thread t takes butterflies t, t + T, ... (the transform index varies fastest).  Every stage
// reads, waits at a barrier, then writes over its inputs.
template <class L, int N, int NF, int T, int NS>
__device__ __forceinline__ void fft_stages(float* s, const float2* tws) {
    if constexpr (NS < N) {
        constexpr int REM = N / NS;
        constexpr int R = (REM % 16 == 0) ? 16 : (REM % 8 == 0) ? 8 : (REM % 4 == 0) ? 4
                        : (REM % 2 == 0) ? 2 : 5;
        static_assert(REM % R == 0, "lengths of the form 2^a 5^b");
        constexpr int NJ = N / R;                 // butterflies per transform
        constexpr int NB = NJ * NF;               // butterflies per stage
        constexpr int PER = (NB + T - 1) / T;     // butterflies per thread
        float2 v[PER][R];
#pragma unroll
        for (int b = 0; b < PER; ++b) {
            const int idx = threadIdx.x + b * T;
            if (NB % T == 0 || idx < NB) {
                const int f = idx % NF, j = idx / NF;
#pragma unroll
                for (int r = 0; r < R; ++r) v[b][r] = L::ld(s, f, j + r * NJ);
            }
        }
        __syncthreads();
#pragma unroll
        for (int b = 0; b < PER; ++b) {
            const int idx = threadIdx.x + b * T;
            if (NB % T == 0 || idx < NB) {
                const int f = idx % NF, j = idx / NF;
                const int k = j % NS;
                if constexpr (NS > 1) {
                    // odd powers from the table, even ones as squares of lower powers
                    float2 w[R];
#pragma unroll
                    for (int r = 1; r < R; ++r)
                        w[r] = (r & 1) ? twiddle<N>(tws, k * r * (N / (NS * R))) : cmul(w[r / 2], w[r / 2]);
#pragma unroll
                    for (int r = 1; r < R; ++r) v[b][r] = cmul(v[b][r], w[r]);
                }
                dft<R>(v[b]);
                const int base = (j / NS) * NS * R + k;
#pragma unroll
                for (int r = 0; r < R; ++r) L::st(s, f, base + r * NS, v[b][r]);
            }
        }
        __syncthreads();
        fft_stages<L, N, NF, T, NS * R>(s, tws);
    }
}

// c_k of the orthonormal DCT basis, P[i][k] = c_k cos(pi k (2i+1) / 2N).
template <int N>
__device__ __forceinline__ float dct_c(int k) {
    return k == 0 ? __fsqrt_rn(1.f / (float)N) : __fsqrt_rn(2.f / (float)N);
}

// DCT-II coefficients X_k of the two real sequences packed in the transform Z (a: real part,
// b: imaginary part), from Z_k and Z_{N-k}; t = exp(-i pi k / 2N), c = c_k (times any scale).
__device__ __forceinline__ void dct2_coeffs(float2 Z, float2 Zc, float2 t, float c, float& xa,
                                            float& xb) {
    const float var = 0.5f * (Z.x + Zc.x), vai = 0.5f * (Z.y - Zc.y);   // spectrum of a
    const float vbr = 0.5f * (Z.y + Zc.y), vbi = -0.5f * (Z.x - Zc.x);  // spectrum of b
    xa = c * (t.x * var - t.y * vai);
    xb = c * (t.x * vbr - t.y * vbi);
}

// Spectrum V_k of the reordered sequence whose DCT-III has coefficients Y (already multiplied by
// c_k): V_k = exp(i pi k / 2N) (Y_k - i Y_{N-k}) sk, sk = 1 at k = 0 (Y_N = 0) and 1/2 else.
__device__ __forceinline__ float2 dct3_spec(float yk, float yp, float2 t, float sk) {
    return make_float2((t.x * yk - t.y * yp) * sk, (-t.x * yp - t.y * yk) * sk);
}

// conj(Va + i Vb): the packed spectrum of two real sequences, conjugated so that a forward FFT
// followed by a conjugation evaluates the inverse sum without a 1/N factor.
__device__ __forceinline__ float2 pack_conj(float2 va, float2 vb) {
    return make_float2(va.x - vb.y, -(va.y + vb.x));
}

// Writes transform f's conjugated packed spectra at slots k and N-k (0 <= k <= N/2) from the
// DCT-III coefficients (times c) of both sequences at k and at N-k; t = exp(-i pi k / 2N).
// The spectrum of a real sequence is Hermitian, so slot N-k takes the conjugates of slot k's
// two spectra: one complex product per sequence serves both slots.
template <class L, int N>
__device__ __forceinline__ void inv_pair(float* s, int f, int k, float ya_k, float yb_k, float ya_p,
                                         float yb_p, float2 t) {
    if (k == 0) {   // V_0 = Y_0 (Y_N = 0)
        L::st(s, f, 0, make_float2(ya_k, -yb_k));
        return;
    }
    const float2 pa = dct3_spec(ya_k, ya_p, t, 0.5f), pb = dct3_spec(yb_k, yb_p, t, 0.5f);
    L::st(s, f, k, pack_conj(pa, pb));
    if (k != N - k) L::st(s, f, N - k, make_float2(pa.x + pb.y, pa.y - pb.x));
}

// Rows of 16000 and 16384 elements (below, quads): one pair of rows a block, one thread per radix-16
// butterfly of its transform.
template <int N>
struct RowCfg {
    static_assert(N == 16000 || N == 16384, "the others run quads");
    static constexpr int NF = 1;
    static constexpr int T = (N * NF / 16 + 31) / 32 * 32;   // whole warps
    using L = PairL<N, NF>;
    static constexpr size_t SMEM = (size_t)L::FLOATS * sizeof(float) + TwN<N>::PADDED * sizeof(float2);
    static constexpr int WANT = 4;          // blocks per SM the carve-out is sized for
};
// ---- rows, forward: T[i][k] = tau * sum_j r_U[i][j] P_M[j][k] ---------------------------------
template <int N>
__global__ void __launch_bounds__(RowCfg<N>::T, 1024 / RowCfg<N>::T)
k_fftdct_rows_fwd(const float* __restrict__ R, float* __restrict__ Tout, int H, int ld, float tau,
                  const float2* __restrict__ tw, const float2* __restrict__ tt, const DevState* st,
                  int skip_if_done) {
    using C = RowCfg<N>;
    using L = typename C::L;
    constexpr int NF = C::NF, T = C::T, Q = N / 4;
    if (skip_if_done && st->done) return;
    extern __shared__ __align__(16) float sm[];
    float2* tws = reinterpret_cast<float2*>(sm + L::FLOATS);
    load_twiddles<N, T>(tws, tw);
    const int row0 = blockIdx.x * 2 * NF;
    // up to four 16-byte pieces of each of the two rows a thread (all loads first), every element
    // stored straight to its slot of the even/odd reordering
    static_assert(NF * Q <= 4 * T, "four pieces per thread at most");
    float4 va[4], vb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int it = threadIdx.x + u * T;
        const int f = it / Q, n = (it % Q) * 4;
        const int ra = row0 + 2 * f, rb = ra + 1;
        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const bool in = it < NF * Q;
        va[u] = in && ra < H ? __ldg(reinterpret_cast<const float4*>(R + (size_t)ra * ld + n)) : z4;
        vb[u] = in && rb < H ? __ldg(reinterpret_cast<const float4*>(R + (size_t)rb * ld + n)) : z4;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int it = threadIdx.x + u * T;
        if (NF * Q < 4 * T && it >= NF * Q) continue;
        const int f = it / Q, n = (it % Q) * 4;
        L::st(sm, f, reorder_pos<N>(n), make_float2(va[u].x, vb[u].x));
        L::st(sm, f, reorder_pos<N>(n + 1), make_float2(va[u].y, vb[u].y));
        L::st(sm, f, reorder_pos<N>(n + 2), make_float2(va[u].z, vb[u].z));
        L::st(sm, f, reorder_pos<N>(n + 3), make_float2(va[u].w, vb[u].w));
    }
    __syncthreads();
    fft_stages<L, N, NF, T, 1>(sm, tws);
    for (int it = threadIdx.x; it < NF * Q; it += T) {
        const int f = it / Q, k0 = (it % Q) * 4;
        const int ra = row0 + 2 * f, rb = ra + 1;
        float xa[4], xb[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int k = k0 + c;
            dct2_coeffs(L::ld(sm, f, k), L::ld(sm, f, (k == 0 ? 0 : N - k)), __ldg(&tt[k]),
                        dct_c<N>(k) * tau, xa[c], xb[c]);
        }
        if (ra < H)
            *reinterpret_cast<float4*>(Tout + (size_t)ra * ld + k0) = make_float4(xa[0], xa[1], xa[2], xa[3]);
        if (rb < H)
            *reinterpret_cast<float4*>(Tout + (size_t)rb * ld + k0) = make_float4(xb[0], xb[1], xb[2], xb[3]);
    }
}

// ---- rows, inverse: z_U[i][j] = sum_k T[i][k] P_M[j][k] --------------------------------------
template <int N>
__global__ void __launch_bounds__(RowCfg<N>::T, 1024 / RowCfg<N>::T)
k_fftdct_rows_inv(const float* __restrict__ Tin, float* __restrict__ Z, int H, int ld,
                  const float2* __restrict__ tw, const float2* __restrict__ tt, const DevState* st,
                  int skip_if_done) {
    using C = RowCfg<N>;
    using L = typename C::L;
    constexpr int NF = C::NF, T = C::T, Q = N / 4;
    if (skip_if_done && st->done) return;
    extern __shared__ __align__(16) float sm[];
    float2* tws = reinterpret_cast<float2*>(sm + L::FLOATS);
    load_twiddles<N, T>(tws, tw);
    const int row0 = blockIdx.x * 2 * NF;
    static_assert(NF * Q <= 4 * T, "four pieces per thread at most");
    float4 va[4], vb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int it = threadIdx.x + u * T;
        const int f = it / Q, k = (it % Q) * 4;
        const int ra = row0 + 2 * f, rb = ra + 1;
        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const bool in = it < NF * Q;
        va[u] = in && ra < H ? *reinterpret_cast<const float4*>(Tin + (size_t)ra * ld + k) : z4;
        vb[u] = in && rb < H ? *reinterpret_cast<const float4*>(Tin + (size_t)rb * ld + k) : z4;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int it = threadIdx.x + u * T;
        if (NF * Q < 4 * T && it >= NF * Q) continue;
        const int f = it / Q, k = (it % Q) * 4;
        L::st(sm, f, k, make_float2(va[u].x, vb[u].x));
        L::st(sm, f, k + 1, make_float2(va[u].y, vb[u].y));
        L::st(sm, f, k + 2, make_float2(va[u].z, vb[u].z));
        L::st(sm, f, k + 3, make_float2(va[u].w, vb[u].w));
    }
    __syncthreads();
    constexpr int NK = N / 2 + 1;
    for (int it = threadIdx.x; it < NF * NK; it += T) {
        const int f = it % NF, k = it / NF;
        const int kc = (k == 0 ? 0 : N - k);
        const float2 xk = L::ld(sm, f, k), xc = L::ld(sm, f, kc);
        const float ck = dct_c<N>(k), cc = dct_c<N>(kc);
        inv_pair<L, N>(sm, f, k, ck * xk.x, ck * xk.y, cc * xc.x, cc * xc.y, __ldg(&tt[k]));
    }
    __syncthreads();
    fft_stages<L, N, NF, T, 1>(sm, tws);
    for (int it = threadIdx.x; it < NF * Q; it += T) {
        const int f = it / Q, n = (it % Q) * 4;
        const int ra = row0 + 2 * f, rb = ra + 1;
        const float2 v0 = L::ld(sm, f, reorder_pos<N>(n)), v1 = L::ld(sm, f, reorder_pos<N>(n + 1));
        const float2 v2 = L::ld(sm, f, reorder_pos<N>(n + 2)), v3 = L::ld(sm, f, reorder_pos<N>(n + 3));
        if (ra < H)
            *reinterpret_cast<float4*>(Z + (size_t)ra * ld + n) = make_float4(v0.x, v1.x, v2.x, v3.x);
        if (rb < H)
            *reinterpret_cast<float4*>(Z + (size_t)rb * ld + n) = make_float4(-v0.y, -v1.y, -v2.y, -v3.y);
    }
}

// rho = r_U^T z_U + r_V^T z_V, the ratio beta and the breakdown test (Alg. 2), by one thread.
__device__ __forceinline__ void finish_rho_fft(DevState* st, double rho_u, int flexible) {
    const double rho_new = rho_u + st->rz_v;
    if (!(rho_new > 0.0) || !isfinite(rho_new)) {
        // rho <= 0 is a breakdown unless the residual is already at the accuracy rounding
        // allows (relative 1e-3 and below)
        if (st->rel > 1e-3 || !isfinite(rho_new)) st->status |= ST_BREAKDOWN;
        st->done = 1;
    } else if (st->p_fresh) {
        st->rho = rho_new;
        st->beta = 0.0;
    } else {
        const double num = flexible ? rho_new - st->rz_old : rho_new;
        st->beta = num / st->rho;
        st->rho = rho_new;
    }
}

// ---- quads: four real sequences as two packed complex transforms ------------------------------
// Lengths to 8192 run four sequences x0 .. x3 (rows, or columns) at a time: the transforms
// x0 + i x2 and x1 + i x3, element m of both in one 16-byte row (x0, x1, x2, x3) of shared memory.
// A thread takes the same butterfly of both: the real parts are one f32x2 pair and the imaginary
// parts another, so every addition and multiplication is one packed instruction for the two,
// multiplying by -i is free, one twiddle and one address serve both, and a stage moves 16 bytes an
// instruction.  The kernels are bound by instruction issue, so that is what counts: about 10
// instructions a complex point and stage, where one transform a thread took 31 (40 % of them
// addresses).  Twiddles come from per-stage tables [r - 1][k] through L1 (consecutive lanes,
// consecutive entries; no products).  Stages are radix 16 (then 8, 4 or 2), or 20 and 10 for the
// 2^a 5^3 lengths (20 = 4 x 5 by the Chinese remainder map, without inner twiddles).  A row of
// padding after every 16 (20) puts the first stage's writes on distinct banks and keeps every
// access of a stage at a fixed offset from the thread's first.  The first stage takes its inputs
// straight from global memory and the last one's outputs go straight there.  Per application
// (caller's arrays, us; one transform a thread before -> quads): 1024^2 47 -> 23, 2048^2 97 -> 44,
// 4096^2 187 -> 159, 8192^2 1277 -> 773, 4000 x 8000 684 -> 438 (the first two and last two with the
// plane copies of the time); with dependent launches and the 2^a 5^3 columns' twiddles in shared
// memory 4096^2 153, 8192^2 768, 4000 x 8000 416.  At 4096^2 the rows take 32 and 42 us and the
// columns 84 (ncu) against 20 each for their bytes: shared-memory and L1 wavefronts fill 60 % of the
// cycles, and 16 warps an SM (128 registers) leave the barriers of the stages exposed.
typedef unsigned long long u64;
struct Cq { u64 re, im; };   // two complex values: (re0, re1), (im0, im1)

__device__ __forceinline__ u64 pk(float a, float b) {
    u64 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ u64 pk(float a) { return pk(a, a); }
__device__ __forceinline__ float2 un(u64 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ u64 padd(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 psub(u64 a, u64 b) {
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 pmul(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 pfma(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 pneg(u64 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ Cq qadd(Cq a, Cq b) { return {padd(a.re, b.re), padd(a.im, b.im)}; }
__device__ __forceinline__ Cq qsub(Cq a, Cq b) { return {psub(a.re, b.re), psub(a.im, b.im)}; }
// a - i b and a + i b
__device__ __forceinline__ Cq qsubi(Cq a, Cq b) { return {padd(a.re, b.im), psub(a.im, b.re)}; }
__device__ __forceinline__ Cq qaddi(Cq a, Cq b) { return {psub(a.re, b.im), padd(a.im, b.re)}; }
// a (x + i y) with the same factor for both
__device__ __forceinline__ Cq qmul(Cq a, float x, float y) {
    const u64 c = pk(x), s = pk(y), n = pk(-y);
    return {pfma(a.im, n, pmul(a.re, c)), pfma(a.re, s, pmul(a.im, c))};
}

template <int R>
__device__ __forceinline__ void qdft(Cq* v);
template <>
__device__ __forceinline__ void qdft<2>(Cq* v) {
    const Cq a = v[0], b = v[1];
    v[0] = qadd(a, b);
    v[1] = qsub(a, b);
}
template <>
__device__ __forceinline__ void qdft<4>(Cq* v) {
    const Cq s02 = qadd(v[0], v[2]), d02 = qsub(v[0], v[2]);
    const Cq s13 = qadd(v[1], v[3]), d13 = qsub(v[1], v[3]);
    v[0] = qadd(s02, s13);
    v[2] = qsub(s02, s13);
    v[1] = qsubi(d02, d13);
    v[3] = qaddi(d02, d13);
}
// * exp(-i pi / 4) and * exp(-3 i pi / 4)
__device__ __forceinline__ Cq qrot1(Cq a) {
    const u64 c = pk(kR2);
    return {pmul(padd(a.re, a.im), c), pmul(psub(a.im, a.re), c)};
}
__device__ __forceinline__ Cq qrot3(Cq a) {
    return {pmul(psub(a.im, a.re), pk(kR2)), pmul(padd(a.re, a.im), pk(-kR2))};
}
template <>
__device__ __forceinline__ void qdft<8>(Cq* v) {
    Cq e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    qdft<4>(e);
    qdft<4>(o);
    o[1] = qrot1(o[1]);
    o[3] = qrot3(o[3]);
    v[0] = qadd(e[0], o[0]);
    v[4] = qsub(e[0], o[0]);
    v[1] = qadd(e[1], o[1]);
    v[5] = qsub(e[1], o[1]);
    v[2] = qsubi(e[2], o[2]);
    v[6] = qaddi(e[2], o[2]);
    v[3] = qadd(e[3], o[3]);
    v[7] = qsub(e[3], o[3]);
}
// 4 x 4 as dft<16> above
template <>
__device__ __forceinline__ void qdft<16>(Cq* v) {
    Cq y[4][4];
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) {
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) y[n1][k2] = v[n1 + 4 * k2];
        qdft<4>(y[n1]);
    }
    y[1][1] = qmul(y[1][1], kC8, -kS8);
    y[1][2] = qrot1(y[1][2]);
    y[1][3] = qmul(y[1][3], kS8, -kC8);
    y[2][1] = qrot1(y[2][1]);
    y[2][2] = {y[2][2].im, pneg(y[2][2].re)};
    y[2][3] = qrot3(y[2][3]);
    y[3][1] = qmul(y[3][1], kS8, -kC8);
    y[3][2] = qrot3(y[3][2]);
    y[3][3] = qmul(y[3][3], -kC8, kS8);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) {
        Cq c[4] = {y[0][k2], y[1][k2], y[2][k2], y[3][k2]};
        qdft<4>(c);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) v[k2 + 4 * k1] = c[k1];
    }
}
// Length 5 as dft<5> above.
template <>
__device__ __forceinline__ void qdft<5>(Cq* v) {
    const Cq t1 = qadd(v[1], v[4]), t2 = qadd(v[2], v[3]);
    const Cq t3 = qsub(v[1], v[4]), t4 = qsub(v[2], v[3]);
    const u64 c1 = pk(kC51), c2 = pk(kC52), s1 = pk(kS51), s2 = pk(kS52);
    const Cq a1 = {pfma(c2, t2.re, pfma(c1, t1.re, v[0].re)), pfma(c2, t2.im, pfma(c1, t1.im, v[0].im))};
    const Cq a2 = {pfma(c1, t2.re, pfma(c2, t1.re, v[0].re)), pfma(c1, t2.im, pfma(c2, t1.im, v[0].im))};
    const Cq b1 = {pfma(s2, t4.re, pmul(s1, t3.re)), pfma(s2, t4.im, pmul(s1, t3.im))};
    const u64 m1 = pk(-kS51);
    const Cq b2 = {pfma(m1, t4.re, pmul(s2, t3.re)), pfma(m1, t4.im, pmul(s2, t3.im))};
    v[0] = qadd(v[0], qadd(t1, t2));
    v[1] = qsubi(a1, b1);
    v[4] = qaddi(a1, b1);
    v[2] = qsubi(a2, b2);
    v[3] = qaddi(a2, b2);
}
// A x 5 with A = 2 or 4, coprime: input n = (5 n1 + A n2) mod 5A, output k = k1 mod A, k2 mod 5.
template <int A>
__device__ __forceinline__ void qdft_x5(Cq* v) {
    constexpr int N = 5 * A, K2 = A == 4 ? 16 : 6;   // K2 = 1 mod 5, 0 mod A
    Cq y[A][5];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
#pragma unroll
        for (int n2 = 0; n2 < 5; ++n2) y[n1][n2] = v[(5 * n1 + A * n2) % N];
        qdft<5>(y[n1]);
    }
#pragma unroll
    for (int k2 = 0; k2 < 5; ++k2) {
        Cq c[A];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) c[n1] = y[n1][k2];
        qdft<A>(c);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[(5 * k1 + K2 * k2) % N] = c[k1];
    }
}
template <>
__device__ __forceinline__ void qdft<10>(Cq* v) { qdft_x5<2>(v); }
template <>
__device__ __forceinline__ void qdft<20>(Cq* v) { qdft_x5<4>(v); }

// Radix of the stage whose sub-transforms have length NS.
__host__ __device__ constexpr int quad_radix(int N, int NS) {
    const int rem = N / NS;
    if (N % 5 == 0) return rem == 100 ? 10 : rem % 20 == 0 ? 20 : rem;
    return rem % 16 == 0 ? 16 : rem;
}
// Shape of a quad launch: GQ quads a block, one thread per first-stage butterfly of a quad; with
// TWS the stages' twiddles lie in shared memory behind the quads.
template <int N, int GQ_, bool TWS_ = false>
struct QuadShape {
    static constexpr int GQ = GQ_;
    static constexpr int PADB = N % 5 == 0 ? 20 : 16;
    static constexpr int T = (N / quad_radix(N, 1) * GQ + 31) / 32 * 32;
    static constexpr int ROWS = N + N / PADB;             // 16-byte rows of a quad
    static constexpr bool TWS = TWS_;
    static constexpr int TWN = N - quad_radix(N, 1);      // twiddles of all stages
    static constexpr size_t SMEM = (size_t)ROWS * GQ * 16 + (TWS ? TWN * sizeof(float2) : 0);
    static constexpr int MINB = 512 / T < 1 ? 1 : (512 / T > 8 ? 8 : 512 / T);
    // the last stage: its sub-transform length, radix and butterflies a thread
    static constexpr int last_ns() {
        int ns = 1;
        while (ns * quad_radix(N, ns) < N) ns *= quad_radix(N, ns);
        return ns;
    }
    static constexpr int LNS = last_ns(), LR = N / LNS;
    static constexpr int LPER = (LNS * GQ + T - 1) / T;
    __device__ static __forceinline__ int slot(int m) { return m + m / PADB; }
};
// Rows: enough threads a block at short lengths.  Columns: at least two quads (a whole 32-byte
// sector of each image row) where they fit shared memory: 4096^2 159 us an application, 165 with
// one quad and two blocks an SM; 2048^2 44 against 48.  The 2^a 5^3 columns take their twiddles from
// shared memory: one block an SM leaves room for them, while in L1 the image's sectors drive them out
// (a fifth of its reads hit): columns of 4000 x 8000 212 to 198 us, of 8000 x 4000 260 to 233, of
// 4000^2 with the rows 212 to 207.  The powers of two lose by it (4096^2 84 to 90, 8192^2 399 to
// 525), 2000 gains nothing (27.5 to 27.9), and rows lose (8000 x 4000 92 to 98).
template <int N>
using RowQ = QuadShape<N, N >= 1000 ? 1 : N >= 512 ? 2 : N >= 256 ? 4 : 8>;
template <int N>
using ColQ = QuadShape<N, N >= 5000 ? 1 : N >= 1000 ? 2 : N >= 512 ? 4 : 8, N % 5 == 0 && N >= 4000>;
constexpr int kQuadMaxN = 8192;
// Lengths whose first stage loads its inputs itself; a radix-20 butterfly has no registers left for
// the addresses, so the 2^a 5^3 lengths bring theirs in through shared memory.
__host__ __device__ constexpr bool quad_direct(int N) { return N % 5 != 0; }

// 16-byte asynchronous global -> shared copy; with `fill` false the 16 bytes are zeros.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool fill) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    const int n = fill ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(n)
                 : "memory");
}

__device__ __forceinline__ Cq qld(const float4* p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return {v.x, v.y};
}
__device__ __forceinline__ void qst(float4* p, Cq v) {
    *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.re, v.im);
}
// The stages' twiddles as quad_stages takes them: in shared memory behind the quads (asynchronous
// copies, complete at the cp.async.wait_all and barrier before the first stage) or where they are.
template <class C>
__device__ __forceinline__ const float2* stage_twiddles(float4* sq, const float2* __restrict__ tw) {
    if constexpr (C::TWS) {
        static_assert(C::TWN % 2 == 0, "whole 16-byte pieces");
        float4* t = sq + C::ROWS * C::GQ;
        for (int e = threadIdx.x; e < C::TWN / 2; e += C::T) cp_async16(t + e, tw + 2 * e, true);
        return reinterpret_cast<const float2*>(t);
    } else {
        return tw;
    }
}
struct FromShared {};   // the first stage's inputs are in the block's rows

// Stockham stages from sub-transform length NS on, in the block's rows s (tw: this stage's table).
// The first stage takes its inputs from `first(q, j, r, NJ)` = element j + r NJ of quad q; the last
// leaves its outputs in `o`: o[b][r] is element j + r LNS of quad q for b's (q, j).  So neither the
// loads nor the stores of a transform pass through shared memory.
template <int N, class C, int NS, class First>
__device__ __forceinline__ void quad_stages(float4* s, const float2* tw, First first,
                                            Cq (&o)[C::LPER][C::LR]) {
    constexpr int R = quad_radix(N, NS), NJ = N / R, NB = NJ * C::GQ, T = C::T;
    constexpr int PER = (NB + T - 1) / T, GQ = C::GQ;
    constexpr bool LAST = NS * R == N;
    constexpr bool SHARED = NS > 1 || std::is_same<First, FromShared>::value;
    // offsets of element r from the first: fixed where the padding advances evenly
    constexpr bool EVEN = NJ % C::PADB == 0;
    Cq v[PER][R];
#pragma unroll
    for (int b = 0; b < PER; ++b) {
        const int idx = threadIdx.x + b * T, q = idx % GQ, j = idx / GQ;
        if (NB % T == 0 || idx < NB) {
            const float4* p = s + C::slot(j) * GQ + q;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if constexpr (SHARED)
                    v[b][r] = qld(EVEN ? p + r * (NJ + NJ / C::PADB) * GQ
                                       : s + C::slot(j + r * NJ) * GQ + q);
                else
                    v[b][r] = first(q, j, r, NJ);
            }
        }
    }
    if constexpr (SHARED && !LAST) __syncthreads();
#pragma unroll
    for (int b = 0; b < PER; ++b) {
        const int idx = threadIdx.x + b * T, q = idx % GQ, j = idx / GQ;
        if (NB % T == 0 || idx < NB) {
            const int k = j % NS;
            if constexpr (NS > 1) {
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    const float2* p = &tw[(r - 1) * NS + k];
                    const float2 w = C::TWS ? *p : __ldg(p);
                    v[b][r] = qmul(v[b][r], w.x, w.y);
                }
            }
            qdft<R>(v[b]);
            if constexpr (LAST) {
#pragma unroll
                for (int r = 0; r < R; ++r) o[b][r] = v[b][r];
            } else {
                const int base = (j / NS) * NS * R + k;
                float4* p = s + C::slot(base) * GQ + q;
                // NS = 1: base is a multiple of PADB = R; else NS is a multiple of PADB
                constexpr int STEP = NS == 1 ? 1 : NS + NS / C::PADB;
                static_assert(NS == 1 ? R == C::PADB : NS % C::PADB == 0, "");
#pragma unroll
                for (int r = 0; r < R; ++r) qst(p + r * STEP * GQ, v[b][r]);
            }
        }
    }
    if constexpr (!LAST) {
        __syncthreads();
        quad_stages<N, C, NS * R>(s, NS > 1 ? tw + (R - 1) * NS : tw, first, o);
    }
}

// Runs f(element of o, q, k) over the last stage's outputs.
template <class C, class F>
__device__ __forceinline__ void quad_outputs(Cq (&o)[C::LPER][C::LR], F f) {
    constexpr int NB = C::LNS * C::GQ;
#pragma unroll
    for (int b = 0; b < C::LPER; ++b) {
        const int idx = threadIdx.x + b * C::T, q = idx % C::GQ, j = idx / C::GQ;
        if (NB % C::T == 0 || idx < NB) {
#pragma unroll
            for (int r = 0; r < C::LR; ++r) f(o[b][r], q, j, r);
        }
    }
}

// Position of element j + r NJ (NJ R = N, R even: the half is known from r) of the even/odd
// reordered sequence in the sequence itself.
template <int N, int R>
__device__ __forceinline__ int source_of(int j, int r, int NJ) {
    return r < R / 2 ? 2 * j + 2 * r * NJ : 2 * N - 1 - 2 * j - 2 * r * NJ;
}

// Coefficients of the four sequences (c times the DCT-II) at k, from Z_k and Z_{N-k}:
// t = exp(-i pi k / 2N); (x0, x1) and (x2, x3).
__device__ __forceinline__ void quad_coeffs(Cq Z, Cq Zc, float2 t, float c, u64& a, u64& b) {
    const u64 tx = pk(0.5f * c * t.x), ty = pk(0.5f * c * t.y), ny = pk(-0.5f * c * t.y);
    a = pfma(psub(Z.im, Zc.im), ny, pmul(padd(Z.re, Zc.re), tx));
    b = pfma(psub(Z.re, Zc.re), ty, pmul(padd(Z.im, Zc.im), tx));
}
// Conjugated packed spectra at slots k and N-k from the DCT-III coefficients (times c) at k and
// at N-k (y*: the sequences x0, x1; z*: x2, x3), as inv_pair above.
__device__ __forceinline__ void quad_inverse(u64 yk, u64 zk, u64 yp, u64 zp, float2 t, Cq& vk,
                                             Cq& vc) {
    const u64 tx = pk(0.5f * t.x), nx = pk(-0.5f * t.x), ny = pk(-0.5f * t.y);
    const u64 ar = pfma(yp, ny, pmul(yk, tx)), ai = pfma(yk, ny, pmul(yp, nx));
    const u64 br = pfma(zp, ny, pmul(zk, tx)), bi = pfma(zk, ny, pmul(zp, nx));
    vk = {psub(ar, bi), pneg(padd(ai, br))};
    vc = {padd(ar, bi), psub(ai, br)};
}

// ---- rows, forward (quads): T[i][k] = tau * sum_j r_U[i][j] P_M[j][k] ------------------------
template <int N>
__global__ void __launch_bounds__(RowQ<N>::T, RowQ<N>::MINB)
k_fftq_rows_fwd(const float* R, float* __restrict__ Tout, int H, int ld, float tau,
                const float2* __restrict__ tw, const float2* __restrict__ tt, const DevState* st,
                int skip_if_done) {
    using C = RowQ<N>;
    constexpr int GQ = C::GQ;
    pdl_enter();
    if (skip_if_done && st->done) return;
    extern __shared__ __align__(16) float4 sq[];
    const int row0 = blockIdx.x * 4 * GQ;                // H is a multiple of 4
    Cq o[C::LPER][C::LR];
    if constexpr (quad_direct(N)) {
        quad_stages<N, C, 1>(sq, tw, [&](int q, int j, int r, int NJ) {
            // (planes hold less than 2^31 elements: 32-bit offsets from a uniform base)
            const unsigned e = (unsigned)min(row0 + 4 * q, H - 4) * ld +
                               source_of<N, quad_radix(N, 1)>(j, r, NJ);
            return Cq{pk(R[e], R[e + ld]), pk(R[e + 2u * ld], R[e + 3u * ld])};
        }, o);
    } else {
        // four columns of four rows a thread, transposed into the rows of the even/odd reordering
        for (int it = threadIdx.x; it < GQ * (N / 4); it += C::T) {
            const int q = it % GQ, n = (it / GQ) * 4;
            const unsigned e = (unsigned)min(row0 + 4 * q, H - 4) * ld + n;
            float4 x[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) x[c] = *reinterpret_cast<const float4*>(R + e + c * ld);
            float4* p = sq + q;
            p[C::slot(reorder_pos<N>(n)) * GQ] = make_float4(x[0].x, x[1].x, x[2].x, x[3].x);
            p[C::slot(reorder_pos<N>(n + 1)) * GQ] = make_float4(x[0].y, x[1].y, x[2].y, x[3].y);
            p[C::slot(reorder_pos<N>(n + 2)) * GQ] = make_float4(x[0].z, x[1].z, x[2].z, x[3].z);
            p[C::slot(reorder_pos<N>(n + 3)) * GQ] = make_float4(x[0].w, x[1].w, x[2].w, x[3].w);
        }
        __syncthreads();
        quad_stages<N, C, 1>(sq, tw, FromShared(), o);
    }
    // X_k from Z_k (in registers) and Z_{N-k} (another thread's)
    __syncthreads();
    quad_outputs<C>(o, [&](Cq& z, int q, int j, int r) { qst(sq + C::slot(j + r * C::LNS) * GQ + q, z); });
    __syncthreads();
    quad_outputs<C>(o, [&](Cq& z, int q, int j, int r) {
        const int k = j + r * C::LNS, row = row0 + 4 * q;
        if (row >= H) return;
        u64 a, b;
        quad_coeffs(z, qld(sq + C::slot(k == 0 ? 0 : N - k) * GQ + q), __ldg(&tt[k]),
                    dct_c<N>(k) * tau, a, b);
        const float2 u = un(a), w = un(b);
        const unsigned e = (unsigned)row * ld + k;
        Tout[e] = u.x;
        Tout[e + ld] = u.y;
        Tout[e + 2u * ld] = w.x;
        Tout[e + 3u * ld] = w.y;
    });
}

// ---- columns (quads): forward DCT, division by the eigenvalues, inverse DCT (in place) -------
// Block b owns the 4 GQ columns from 4 GQ b on.
template <int N>
__global__ void __launch_bounds__(ColQ<N>::T, ColQ<N>::MINB)
k_fftq_cols(float* __restrict__ Tio, int W, int ld, float tau, const float* __restrict__ lamN,
            const float* __restrict__ lamM, const float2* __restrict__ tw,
            const float2* __restrict__ tt, DevState* st, double* partials, int reduce_rho,
            int skip_if_done, int flexible) {
    using C = ColQ<N>;
    constexpr int GQ = C::GQ, T = C::T;
    pdl_enter();
    if (skip_if_done && st->done) return;
    extern __shared__ __align__(16) float4 sq[];
    const int q = threadIdx.x % GQ;                      // T is a multiple of GQ
    const int j0 = (blockIdx.x * GQ + q) * 4;
    const bool in = j0 < W;                              // W is a multiple of 4
    const float4 m = in ? __ldg(reinterpret_cast<const float4*>(lamM + j0)) : make_float4(1.f, 1.f, 1.f, 1.f);
    const float2* tws = stage_twiddles<C>(sq, tw);
    static_assert(!C::TWS || !quad_direct(N), "the copies are waited for with the columns'");
    Cq o[C::LPER][C::LR];
    if constexpr (quad_direct(N)) {
        quad_stages<N, C, 1>(sq, tws, [&](int, int j, int r, int NJ) {
            const int i = source_of<N, quad_radix(N, 1)>(j, r, NJ);
            if (!in) return Cq{0ull, 0ull};
            const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(Tio + ((unsigned)i * ld + j0));
            return Cq{x.x, x.y};
        }, o);
    } else {
        for (int it = threadIdx.x; it < GQ * N; it += T) {
            const int i = it / GQ;
            cp_async16(sq + C::slot(reorder_pos<N>(i)) * GQ + q,
                       Tio + ((unsigned)i * ld + (in ? j0 : 0)), in);
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
        quad_stages<N, C, 1>(sq, tws, FromShared(), o);
    }
    __syncthreads();
    quad_outputs<C>(o, [&](Cq& z, int, int j, int r) { qst(sq + C::slot(j + r * C::LNS) * GQ + q, z); });
    __syncthreads();
    CSum part;
    for (int it = threadIdx.x; it < GQ * (N / 2 + 1); it += T) {
        const int k = it / GQ, kc = k == 0 ? 0 : N - k;
        const float2 t = __ldg(&tt[k]);
        const float ck = dct_c<N>(k), cc = dct_c<N>(kc);
        float4* pk_ = sq + C::slot(k) * GQ + q;
        float4* pc_ = sq + C::slot(kc) * GQ + q;
        const Cq Z = qld(pk_), Zc = qld(pc_);
        // w = t V for both sequences of a transform: X_k = c_k Re w, X_{N-k} = -c_{N-k} Im w
        const u64 sr = padd(Z.re, Zc.re), si = padd(Z.im, Zc.im);
        const u64 dr = psub(Z.re, Zc.re), di = psub(Z.im, Zc.im);
        const float hk = 0.5f * ck, hc = 0.5f * cc;
        const float2 xa = un(pfma(di, pk(-hk * t.y), pmul(sr, pk(hk * t.x))));
        const float2 xb = un(pfma(dr, pk(hk * t.y), pmul(si, pk(hk * t.x))));
        const float2 ya = un(pfma(sr, pk(-hc * t.y), pmul(di, pk(-hc * t.x))));
        const float2 yb = un(pfma(si, pk(-hc * t.y), pmul(dr, pk(hc * t.x))));
        const float lk = __ldg(&lamN[k]), lc = __ldg(&lamN[kc]);
        // X / (l + m); the (0, 0) entry (the constant, the Laplacian's null space) is zero (the
        // denominators lie in (0, 8]: the fast division is within 2 ulp)
        const float s0 = (k | j0) != 0 ? __fdividef(xa.x, lk + m.x) : 0.f;
        const float s1 = __fdividef(xa.y, lk + m.y);
        const float s2 = __fdividef(xb.x, lk + m.z), s3 = __fdividef(xb.y, lk + m.w);
        const float p0 = (kc | j0) != 0 ? __fdividef(ya.x, lc + m.x) : 0.f;
        const float p1 = __fdividef(ya.y, lc + m.y);
        const float p2 = __fdividef(yb.x, lc + m.z), p3 = __fdividef(yb.y, lc + m.w);
        if (in) {
            const float a = (xa.x * s0 + xa.y * s1) + (xb.x * s2 + xb.y * s3);
            const float b = (ya.x * p0 + ya.y * p1) + (yb.x * p2 + yb.y * p3);
            part.add(kc != k ? a + b : a);
        }
        if (k == 0) {   // V_0 = Y_0 (Y_N = 0)
            qst(pk_, {pk(ck * s0, ck * s1), pk(-ck * s2, -ck * s3)});
        } else {
            Cq vk, vc;
            quad_inverse(pk(ck * s0, ck * s1), pk(ck * s2, ck * s3), pk(cc * p0, cc * p1),
                         pk(cc * p2, cc * p3), t, vk, vc);
            qst(pk_, vk);
            if (kc != k) qst(pc_, vc);
        }
    }
    __syncthreads();
    quad_stages<N, C, 1>(sq, tws, FromShared(), o);
    if (in)
        quad_outputs<C>(o, [&](Cq& z, int, int j, int r) {
            const int i = source_of<N, C::LR>(j, r, C::LNS);
            const float2 a = un(z.re), b = un(z.im);
            *reinterpret_cast<float4*>(Tio + ((unsigned)i * ld + j0)) = make_float4(a.x, a.y, -b.x, -b.y);
        });
    if (!reduce_rho) return;
    // r_U^T z_U = sum S^2 / (tau (l + m)) (the basis is orthonormal)
    double vv[1] = {part.value() / (double)tau}, tot[1];
    const Blk blk = single_blk();
    if (grid_reduce<1>(vv, partials, &st->counter, tot, blk.nblk, blk.bid) && threadIdx.x == 0)
        finish_rho_fft(st, tot[0], flexible);
}

// ---- rows, inverse (quads): z_U[i][j] = sum_k T[i][k] P_M[j][k] ------------------------------
// The first stage forms its inputs, V_k = exp(i pi k / 2N) (Y_k - i Y_{N-k}) / 2 (V_0 = Y_0) of the
// four rows, from the row itself at k and N-k.
template <int N>
__global__ void __launch_bounds__(RowQ<N>::T, RowQ<N>::MINB)
k_fftq_rows_inv(const float* Tin, float* __restrict__ Z, int H, int ld,
                const float2* __restrict__ tw, const float2* __restrict__ tt, const DevState* st,
                int skip_if_done) {
    using C = RowQ<N>;
    constexpr int GQ = C::GQ;
    pdl_enter();
    if (skip_if_done && st->done) return;
    extern __shared__ __align__(16) float4 sq[];
    const int row0 = blockIdx.x * 4 * GQ;
    Cq o[C::LPER][C::LR];
    quad_stages<N, C, 1>(sq, tw, [&](int q, int j, int r, int NJ) {
        const int k = j + r * NJ;
        const bool zero = r == 0 && j == 0;
        const unsigned row = (unsigned)min(row0 + 4 * q, H - 4) * ld;
        const unsigned p = row + k, n = row + (zero ? 0 : N - k);
        float2 t = __ldg(&tt[k]);
        const float c = dct_c<N>(1);
        // (Y_0 - i 0) sqrt(1/N) without the half: the factor of k = 0
        const float tx = zero ? dct_c<N>(0) : 0.5f * c * t.x, ty = zero ? 0.f : 0.5f * c * t.y;
        const u64 px = pk(tx), nx = pk(zero ? 0.f : -tx), ny = pk(-ty);
        const u64 yk = pk(Tin[p], Tin[p + ld]);
        const u64 zk = pk(Tin[p + 2u * ld], Tin[p + 3u * ld]);
        const u64 yp = pk(Tin[n], Tin[n + ld]);
        const u64 zp = pk(Tin[n + 2u * ld], Tin[n + 3u * ld]);
        const u64 ar = pfma(yp, ny, pmul(yk, px)), ai = pfma(yk, ny, pmul(yp, nx));
        const u64 br = pfma(zp, ny, pmul(zk, px)), bi = pfma(zk, ny, pmul(zp, nx));
        return Cq{psub(ar, bi), pneg(padd(ai, br))};
    }, o);
    quad_outputs<C>(o, [&](Cq& z, int q, int j, int r) {
        const int row = row0 + 4 * q;
        if (row >= H) return;
        const unsigned e = (unsigned)row * ld + source_of<N, C::LR>(j, r, C::LNS);
        const float2 a = un(z.re), b = un(z.im);
        Z[e] = a.x;
        Z[e + ld] = a.y;
        Z[e + 2u * ld] = -b.x;
        Z[e + 3u * ld] = -b.y;
    });
}

// exp(-i pi k / 2N), k < N, and the twiddles exp(-2 pi i m / N) of one transform length, from FP64
// cospi / sinpi.
__global__ void k_build_fft_tables(float2* tw, float2* tt, int N) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < N; k += gridDim.x * blockDim.x) {
        const double a = 2.0 * (double)k / (double)N, b = (double)k / (2.0 * (double)N);
        tw[k] = make_float2((float)cospi(a), (float)-sinpi(a));
        tt[k] = make_float2((float)cospi(b), (float)-sinpi(b));
    }
}

// A quad stage's twiddles: w[(r - 1) NS + k] = exp(-2 pi i k r / (NS R)).
__global__ void k_build_stage_twiddles(float2* w, int NS, int R) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < (R - 1) * NS; e += gridDim.x * blockDim.x) {
        const double a = 2.0 * (double)(e % NS) * (double)(e / NS + 1) / ((double)NS * (double)R);
        w[e] = make_float2((float)cospi(a), (float)-sinpi(a));
    }
}

cudaError_t build_tables(float2* tw, float2* tt, int n) {
    k_build_fft_tables<<<(n + 255) / 256, 256>>>(tw, tt, n);
    if (n <= kQuadMaxN)   // the quads' stages take the twiddles' place
        for (int ns = quad_radix(n, 1); ns < n;) {
            const int r = quad_radix(n, ns);
            k_build_stage_twiddles<<<((r - 1) * ns + 255) / 256, 256>>>(tw, ns, r);
            tw += (r - 1) * ns;
            ns *= r;
        }
    return cudaGetLastError();
}

bool pow2_in(int n, int lo, int hi) { return n >= lo && n <= hi && (n & (n - 1)) == 0; }

// Lengths compiled in besides the powers of two: 2^a 5^3, the sides of the 4000 x M images of the
// paper's size study.
bool row_len_ok(int n) {
    return pow2_in(n, kFftMinN, kFftMaxRowN) || n == 2000 || n == 4000 || n == 8000 || n == 16000;
}
bool col_len_ok(int n) {
    return pow2_in(n, kFftMinN, kFftMaxColN) || n == 2000 || n == 4000 || n == 8000;
}

// Calls f with the length n as a compile-time constant.
template <int N>
struct Len { static constexpr int value = N; };
template <class F>
cudaError_t with_col_len(int n, F f) {
    switch (n) {
        case 64: return f(Len<64>());
        case 128: return f(Len<128>());
        case 256: return f(Len<256>());
        case 512: return f(Len<512>());
        case 1024: return f(Len<1024>());
        case 2048: return f(Len<2048>());
        case 4096: return f(Len<4096>());
        case 8192: return f(Len<8192>());
        case 2000: return f(Len<2000>());
        case 4000: return f(Len<4000>());
        case 8000: return f(Len<8000>());
        default: return cudaErrorInvalidValue;
    }
}
template <class F>
cudaError_t with_row_len(int n, F f) {
    switch (n) {
        case 16384: return f(Len<16384>());
        case 16000: return f(Len<16000>());
        default: return with_col_len(n, f);
    }
}

// Dynamic shared memory of a kernel, and a carve-out that holds `want` blocks per SM (the rest of
// the SM's 256 KB stays L1).  Set once per plan.
template <class K>
cudaError_t prepare(K k, size_t smem, int want) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const size_t per_block = smem + 1024;   // with the per-block reservation
    const int pct = (int)std::min<size_t>(100, (per_block * want * 100 + 228 * 1024 - 1) / (228 * 1024));
    return cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
}

template <int N>
cudaError_t prepare_rows() {
    cudaError_t e;
    if constexpr (N <= kQuadMaxN) {
        using C = RowQ<N>;
        e = prepare(k_fftq_rows_fwd<N>, C::SMEM, C::MINB);
        return e != cudaSuccess ? e : prepare(k_fftq_rows_inv<N>, C::SMEM, C::MINB);
    } else {
        using C = RowCfg<N>;
        e = prepare(k_fftdct_rows_fwd<N>, C::SMEM, C::WANT);
        return e != cudaSuccess ? e : prepare(k_fftdct_rows_inv<N>, C::SMEM, C::WANT);
    }
}

template <int N>
cudaError_t rows_fwd(const float* R, float* Tout, int H, int ld, float tau, const float2* tw,
                     const float2* tt, const DevState* st, int skip, bool pdl, cudaStream_t s) {
    if constexpr (N <= kQuadMaxN) {
        using C = RowQ<N>;
        return launch_kernel(pdl, k_fftq_rows_fwd<N>, (H + 4 * C::GQ - 1) / (4 * C::GQ), C::T,
                             C::SMEM, s, R, Tout, H, ld, tau, tw, tt, st, skip);
    } else {
        using C = RowCfg<N>;
        k_fftdct_rows_fwd<N><<<(H + 2 * C::NF - 1) / (2 * C::NF), C::T, C::SMEM, s>>>(
            R, Tout, H, ld, tau, tw, tt, st, skip);
        return cudaGetLastError();
    }
}

template <int N>
cudaError_t rows_inv(const float* Tin, float* Z, int H, int ld, const float2* tw, const float2* tt,
                     const DevState* st, int skip, bool pdl, cudaStream_t s) {
    if constexpr (N <= kQuadMaxN) {
        using C = RowQ<N>;
        return launch_kernel(pdl, k_fftq_rows_inv<N>, (H + 4 * C::GQ - 1) / (4 * C::GQ), C::T,
                             C::SMEM, s, Tin, Z, H, ld, tw, tt, st, skip);
    } else {
        using C = RowCfg<N>;
        k_fftdct_rows_inv<N><<<(H + 2 * C::NF - 1) / (2 * C::NF), C::T, C::SMEM, s>>>(
            Tin, Z, H, ld, tw, tt, st, skip);
        return cudaGetLastError();
    }
}

template <int N>
int col_blocks(int W) {
    return (W + 4 * ColQ<N>::GQ - 1) / (4 * ColQ<N>::GQ);
}

}  // namespace

bool fft_dct_supported(int H, int W) {
    return col_len_ok(H) && row_len_ok(W);
}

size_t fft_dct_bytes(int H, int W) {
    if (!fft_dct_supported(H, W)) return 0;
    return 2 * ((size_t)H + (size_t)W) * sizeof(float2) + 1024;
}

int fft_dct_max_blocks(int H, int W) {
    if (!fft_dct_supported(H, W)) return 0;
    return (W + 3) / 4;
}

cudaError_t fft_dct_setup(DctPlan& d, char* mem) {
    d.fft_ready = 0;
    if (!fft_dct_supported(d.H, d.W)) return cudaSuccess;
    float2* f = reinterpret_cast<float2*>(mem);
    d.fftTwN = f; f += d.H;
    d.fftTtN = f; f += d.H;
    d.fftTwM = f; f += d.W;
    d.fftTtM = f; f += d.W;
    cudaError_t e = build_tables(d.fftTwN, d.fftTtN, d.H);
    if (e == cudaSuccess) e = build_tables(d.fftTwM, d.fftTtM, d.W);
    if (e == cudaSuccess)
        e = with_col_len(d.H, [](auto n) {
            using C = ColQ<n.value>;
            return prepare(k_fftq_cols<n.value>, C::SMEM, C::MINB);
        });
    if (e == cudaSuccess) e = with_row_len(d.W, [](auto n) { return prepare_rows<n.value>(); });
    if (e == cudaSuccess) d.fft_ready = 1;
    return e;
}

cudaError_t fft_dct_apply(const DctPlan& d, const float* rU, float* zU, int ld, DevState* st,
                          int reduce_rho, const StencilArgs& a, double* partials, int skip_if_done,
                          cudaStream_t s) {
    if (!d.fft_ready) return cudaErrorInvalidValue;
    const int H = d.H, W = d.W;
    float* T = d.T1;
    const bool pdl = a.pdl != 0;
    cudaError_t e = with_row_len(W, [&](auto n) {
        return rows_fwd<n.value>(rU, T, H, ld, d.tau, d.fftTwM, d.fftTtM, st, skip_if_done, pdl, s);
    });
    if (e != cudaSuccess) return e;
    e = with_col_len(H, [&](auto n) {
        using C = ColQ<n.value>;
        return launch_kernel(pdl, k_fftq_cols<n.value>, col_blocks<n.value>(W), C::T, C::SMEM, s, T,
                             W, ld, d.tau, d.lamN, d.lamM, d.fftTwN, d.fftTtN, st, partials,
                             reduce_rho, skip_if_done, a.flexible);
    });
    if (e != cudaSuccess) return e;
    return with_row_len(W, [&](auto n) {
        return rows_inv<n.value>(T, zU, H, ld, d.fftTwM, d.fftTtM, st, skip_if_done, pdl, s);
    });
}

}  // namespace irls
