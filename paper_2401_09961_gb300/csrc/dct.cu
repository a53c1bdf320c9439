// Laplacian block of the preconditioner (Sec. 3.3 of arXiv 2401.09961):
//   S^T S Z + Z T T^T = tau R   solved as   Z = P_S [ (P_S^T tau R P_T) / (l_i + m_j) ] P_T^T
// with the zero-frequency coefficient set to 0 (the pseudo-inverse choice of Appendix B).
// P_S, P_T are the orthonormal DCT-II eigenvector matrices of the 1-D Neumann Laplacians, built
// once per plan from the closed form P[i][k] = c_k cos(pi k (2i+1) / 2N).
//
// Float32 products on the CUDA cores, in even / odd folded form.  P[n-1-i][k] = (-1)^k P[i][k], so
// folding the image along both sides splits the map into four independent quadrants (s: parity
// of the row frequency k, q: of the column frequency l), each a chain of half-size products
// (half the multiply-adds of the full-size ones; the middle entry of an odd side is its own
// mirror and counts once):
//   fold     Q_sq[i'][j'] = R[i'][j'] +- R[H-1-i'][j'] +- (R[i'][W-1-j'] +- R[H-1-i'][W-1-j'])
//   stage 1  T_sq[j'][a]  = sum_i' Q_sq[i'][j'] PN[i'][2a+s]
//   stage 2  G_sq[a][b]   = tau sum_j' T_sq[j'][a] PM[j'][2b+q] / (l_k + m_l), (0, 0) -> 0;
//            rho_U        = sum F G over the spectrum (= r_U^T z_U, Parseval)
//   stage 3  Y_sq[b][i']  = sum_a G_sq[a][b] PN[i'][2a+s]
//   stage 4  Z_sq[i'][j'] = sum_b Y_sq[b][i'] PM[j'][2b+q]
//   unfold   Z[i'][j'] = sum_sq Z_sq, mirrored rows with the sign of s, columns of q
// Every stage is C[m][n] = sum_k A[k][m] B[k][n] with the rows of both operands contiguous, and
// C is the next stage's A as it lies.
#include <algorithm>

#include "irls_internal.cuh"
#include "reduce.cuh"

namespace irls {

cudaError_t umma_dct_apply(const DctPlan& d, const float* rU, float* zU, int ld, DevState* st,
                           int reduce_rho, const StencilArgs& a, double* partials,
                           int skip_if_done, cudaStream_t s, const float* src, int ld_src);
size_t umma_dct_bytes(int H, int W, int prec);
cudaError_t umma_dct_setup(DctPlan& d, char* mem);
void umma_dct_release(DctPlan& d);
cudaError_t umma_dct_reset(const DctPlan& d, cudaStream_t s);
bool umma_dct_stall(DctPlan& d, int on);

namespace {

__device__ __forceinline__ unsigned long long dup2(float b) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(b));
    return d;
}
__device__ __forceinline__ void fma2(unsigned long long& c, unsigned long long a,
                                     unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

// rho = r_U^T z_U + r_V^T z_V, the ratio beta and the breakdown test (Alg. 2), by one thread.
__device__ __forceinline__ void finish_rho(DevState* st, double rho_u, int flexible) {
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

// One stage over the four quadrants (blockIdx.z = s + 2 q): operands A (quadrant stride sa,
// pitch lda, K x M) and B (its parity's half basis, pitch ldb, K x N), output C (stride sc,
// pitch ldc, M x N).  Pitches are multiples of four floats.
struct QuadArgs {
    const float *A, *B0, *B1;
    float* C;
    size_t sa, sc;
    int lda, ldb, ldc;
    int M, N, K;
    int by_q;               // B's parity: q (stages 2, 4) or s (stages 1, 3)
    int n_k, n_l;           // stage 2: H, W (frequency counts)
    const float *lam_k, *lam_l;
    float scale;            // stage 2: tau
    int rho, flexible;
    DevState* st;
    double* partials;
    int skip_if_done;
    int pdl;                // dependent launch (host)
};

// Tiles.  A thread owns MR x NR outputs (row and column groups of four, spread over the tile);
// KG groups of threads split the k-chunk and are summed at the end.  The chunks come through a
// ring of 16-byte asynchronous copies.  The multiply-adds are packed pairs along the rows
// (fma.rn.f32x2).
//   Large  128 x 128, 16 x 8 a thread: 60.5 TFLOP/s at 4096^2 (of 78 the FMA pipes could do).
//          The shared-memory return path sets the thread tile: a warp's 16-byte load takes four
//          cycles of it, in which the SM issues 16 multiply-adds a lane, so 8 x 8 just balances
//          and 16 x 8 leaves a quarter free.  (Full-size products, 8 x 8 a thread, operands
//          staged through registers, as before: 43 TFLOP/s of twice the work.)
//   Medium  64 x 64, 8 x 8 a thread, four k-groups: 53 TFLOP/s at 4096^2, a quarter of the work
//          a block.  One block's eight warps keep all four schedulers busy.
//   Small   32 x 32, 4 x 4 a thread, four k-groups: for sides where the others leave SMs idle.
template <int MR_, int NR_, int TX_, int TY_, int KG_, int BKG_, int ST_, int MINB_>
struct QuadTile {
    static constexpr int MR = MR_, NR = NR_, TX = TX_, TY = TY_, KG = KG_, BKG = BKG_, ST = ST_,
                         MINB = MINB_;
    static constexpr int RG = MR / 4, CG = NR / 4, G = TX * TY, T = G * KG, BK = BKG * KG;
    static constexpr int BM = MR * TY, BN = NR * TX;
    static constexpr int BUF = BK * (BM + BN);              // floats of one chunk
    static constexpr int RED = (KG - 1) * G * MR * NR;      // floats of the groups' partial sums
    static constexpr int SMEM = (ST * BUF > RED ? ST * BUF : RED) * 4;
    static constexpr int PA = BK * BM / 4, PB = BK * BN / 4;   // 16-byte pieces of a chunk
    static_assert(PA % T == 0 && PB % T == 0, "whole pieces per thread");
};
using TileL = QuadTile<16, 8, 16, 8, 1, 8, 4, 2>;
using TileM = QuadTile<8, 8, 8, 8, 4, 8, 3, 2>;
using TileS = QuadTile<4, 4, 8, 8, 4, 8, 3, 3>;

__device__ __forceinline__ void copy16(float* smem, const float* gmem, bool fill) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    const int n = fill ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(n)
                 : "memory");
}

template <class C, bool SPECTRUM>
__global__ void __launch_bounds__(C::T, C::MINB) k_quad_gemm_f32(QuadArgs f) {
    pdl_enter();
    if (f.skip_if_done && f.st->done) return;
    constexpr int BM = C::BM, BN = C::BN, BK = C::BK, RG = C::RG, CG = C::CG;
    extern __shared__ __align__(16) float sm[];
    const int tid = threadIdx.x, grp = tid / C::G, tg = tid % C::G;
    // a warp's lanes take 8 columns by 4 rows of threads
    const int wg = tg >> 5, lane = tg & 31;
    const int tx = (wg % (C::TX / 8)) * 8 + (lane & 7), ty = (wg / (C::TX / 8)) * 4 + (lane >> 3);
    const int z = blockIdx.z, s = z & 1, q = z >> 1;
    const int m_blk = blockIdx.y * BM, n_blk = blockIdx.x * BN;
    const float* A = f.A + z * f.sa;
    const float* B = (f.by_q ? q : s) ? f.B1 : f.B0;

    auto load = [&](int kt) {
        float* buf = sm + (kt % C::ST) * C::BUF;
        const int k0 = kt * BK;
#pragma unroll
        for (int e = 0; e < C::PA / C::T; ++e) {
            const int p = tid + e * C::T, k = p / (BM / 4), c = (p % (BM / 4)) * 4;
            const bool ok = k0 + k < f.K && m_blk + c < f.lda;
            copy16(buf + k * BM + c, ok ? A + (size_t)(k0 + k) * f.lda + m_blk + c : A, ok);
        }
#pragma unroll
        for (int e = 0; e < C::PB / C::T; ++e) {
            const int p = tid + e * C::T, k = p / (BN / 4), c = (p % (BN / 4)) * 4;
            const bool ok = k0 + k < f.K && n_blk + c < f.ldb;
            copy16(buf + BK * BM + k * BN + c, ok ? B + (size_t)(k0 + k) * f.ldb + n_blk + c : B,
                   ok);
        }
    };

    // acc[g][p][n]: rows 2p, 2p + 1 of row group g packed, column n of the thread
    unsigned long long acc[RG][2][C::NR];
#pragma unroll
    for (int g = 0; g < RG; ++g)
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int n = 0; n < C::NR; ++n) acc[g][p][n] = 0ull;

    const int nk = (f.K + BK - 1) / BK;
#pragma unroll
    for (int t = 0; t < C::ST - 1; ++t) {
        if (t < nk) load(t);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    for (int kt = 0; kt < nk; ++kt) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(C::ST - 2) : "memory");
        __syncthreads();   // chunk kt landed for all; chunk kt - 1 is read by all
        if (kt + C::ST - 1 < nk) load(kt + C::ST - 1);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        const float* ab = sm + (kt % C::ST) * C::BUF + grp * C::BKG * BM + ty * 4;
        const float* bb = sm + (kt % C::ST) * C::BUF + BK * BM + grp * C::BKG * BN + tx * 4;
#pragma unroll
        for (int k = 0; k < C::BKG; ++k) {
            ulonglong2 a[RG];
            float4 b[CG];
#pragma unroll
            for (int g = 0; g < RG; ++g)
                a[g] = *reinterpret_cast<const ulonglong2*>(ab + k * BM + g * (BM / RG));
#pragma unroll
            for (int c = 0; c < CG; ++c)
                b[c] = *reinterpret_cast<const float4*>(bb + k * BN + c * (BN / CG));
#pragma unroll
            for (int c = 0; c < CG; ++c) {
                const unsigned long long bd[4] = {dup2(b[c].x), dup2(b[c].y), dup2(b[c].z),
                                                  dup2(b[c].w)};
#pragma unroll
                for (int g = 0; g < RG; ++g)
#pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        fma2(acc[g][0][4 * c + n], a[g].x, bd[n]);
                        fma2(acc[g][1][4 * c + n], a[g].y, bd[n]);
                    }
            }
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");

    if constexpr (C::KG > 1) {
        // the groups' partial sums, added by the first group in the order of the groups
        constexpr int V2 = RG * 2 * C::NR / 2;   // 16-byte pieces of a thread
        ulonglong2* red = reinterpret_cast<ulonglong2*>(sm);
        __syncthreads();
        if (grp > 0) {
#pragma unroll
            for (int e = 0; e < V2; ++e) {
                const unsigned long long* x = acc[e / C::NR][(e / (C::NR / 2)) % 2] + 2 * (e % (C::NR / 2));
                red[((grp - 1) * V2 + e) * C::G + tg] = make_ulonglong2(x[0], x[1]);
            }
        }
        __syncthreads();
        if (grp == 0) {
#pragma unroll
            for (int g = 1; g < C::KG; ++g)
#pragma unroll
                for (int e = 0; e < V2; ++e) {
                    unsigned long long* x = acc[e / C::NR][(e / (C::NR / 2)) % 2] + 2 * (e % (C::NR / 2));
                    const ulonglong2 y = red[((g - 1) * V2 + e) * C::G + tg];
                    x[0] = add2(x[0], y.x);
                    x[1] = add2(x[1], y.y);
                }
        }
    }

    CSum part;
    if (C::KG == 1 || grp == 0) {
        float* __restrict__ out = f.C + z * f.sc;
#pragma unroll
        for (int g = 0; g < RG; ++g)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int m = m_blk + g * (BM / RG) + ty * 4 + r;
                if (m >= f.M) continue;
#pragma unroll
                for (int c = 0; c < CG; ++c) {
                    const int n0 = n_blk + c * (BN / CG) + tx * 4;
                    if (n0 >= f.ldc) continue;
                    float v[4];
#pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        const float2 x = unpack2(acc[g][r / 2][4 * c + n]);
                        v[n] = r & 1 ? x.y : x.x;
                    }
                    if constexpr (SPECTRUM) {
                        // frequencies k = 2m + s, l = 2n + q: tau v / (l_k + m_l)
                        const int k = 2 * m + s;
                        const float lk = k < f.n_k ? f.lam_k[k] : 0.f;
                        float row = 0.f;
#pragma unroll
                        for (int n = 0; n < 4; ++n) {
                            const int l = 2 * (n0 + n) + q;
                            const bool ok = k < f.n_k && l < f.n_l && (k | l) != 0;
                            const float o = ok ? f.scale * v[n] / (lk + f.lam_l[l]) : 0.f;
                            row += ok ? v[n] * o : 0.f;
                            v[n] = o;
                        }
                        part.add(row);
                    }
                    *reinterpret_cast<float4*>(out + (size_t)m * f.ldc + n0) =
                        make_float4(v[0], v[1], v[2], v[3]);
                }
            }
    }
    if constexpr (SPECTRUM) {
        if (!f.rho) return;
        double vv[1] = {part.value()}, tot[1];
        const unsigned nxy = gridDim.x * gridDim.y;
        if (grid_reduce<1>(vv, f.partials, &f.st->counter, tot, nxy * gridDim.z,
                           blockIdx.x + gridDim.x * blockIdx.y + nxy * z) && tid == 0)
            finish_rho(f.st, tot[0], f.flexible);
    }
}

// Quadrant planes of R (pitch ldr) into Q (four planes hH x ldq): a thread takes four columns of
// a row pair and their mirrors.  Bound by memory: 4 bytes a pixel read and written.
__global__ void __launch_bounds__(256)
k_quad_fold(const float* R, int ldr, int H, int W, float* __restrict__ Q, int ldq, int vec,
            const DevState* st, int skip_if_done) {
    pdl_enter();
    if (skip_if_done && st->done) return;
    const int hH = (H + 1) / 2, hW = (W + 1) / 2;
    const int j0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int i = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= hH || j0 >= ldq) return;
    const float* up = R + (size_t)i * ldr;
    const float* dn = R + (size_t)(H - 1 - i) * ldr;
    float a[4] = {0, 0, 0, 0}, b[4] = {0, 0, 0, 0}, c[4] = {0, 0, 0, 0}, d[4] = {0, 0, 0, 0};
    if (vec && j0 + 3 < hW) {
        const float4 x = *reinterpret_cast<const float4*>(up + j0);
        const float4 y = *reinterpret_cast<const float4*>(dn + j0);
        const float4 u = *reinterpret_cast<const float4*>(up + W - 4 - j0);
        const float4 v = *reinterpret_cast<const float4*>(dn + W - 4 - j0);
        a[0] = x.x; a[1] = x.y; a[2] = x.z; a[3] = x.w;
        b[0] = y.x; b[1] = y.y; b[2] = y.z; b[3] = y.w;
        c[0] = u.w; c[1] = u.z; c[2] = u.y; c[3] = u.x;
        d[0] = v.w; d[1] = v.z; d[2] = v.y; d[3] = v.x;
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (j0 + e < hW) {
                a[e] = up[j0 + e];
                b[e] = dn[j0 + e];
                c[e] = up[W - 1 - j0 - e];
                d[e] = dn[W - 1 - j0 - e];
            }
    }
    float o[4][4];
    const bool mi = 2 * i == H - 1;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const bool mj = 2 * (j0 + e) == W - 1;
        const float se = mi ? a[e] : a[e] + b[e], de = mi ? 0.f : a[e] - b[e];   // column j'
        const float sm = mi ? c[e] : c[e] + d[e], dm = mi ? 0.f : c[e] - d[e];   // its mirror
        o[0][e] = mj ? se : se + sm;
        o[1][e] = mj ? de : de + dm;
        o[2][e] = mj ? 0.f : se - sm;
        o[3][e] = mj ? 0.f : de - dm;
    }
    const size_t plane = (size_t)hH * ldq;
#pragma unroll
    for (int z = 0; z < 4; ++z)
        *reinterpret_cast<float4*>(Q + z * plane + (size_t)i * ldq + j0) =
            make_float4(o[z][0], o[z][1], o[z][2], o[z][3]);
}

// Z (pitch ldz) from its quadrant planes (hH x ldq each).
__global__ void __launch_bounds__(256)
k_quad_unfold(const float* Q, int ldq, int H, int W, float* __restrict__ Z, int ldz,
              int vec, const DevState* st, int skip_if_done) {
    pdl_enter();
    if (skip_if_done && st->done) return;
    const int hH = (H + 1) / 2, hW = (W + 1) / 2;
    const int j0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int i = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= hH || j0 >= hW) return;
    const size_t plane = (size_t)hH * ldq, o = (size_t)i * ldq + j0;
    float a[4], b[4], c[4], d[4];   // (i, j), (H-1-i, j), (i, W-1-j), (H-1-i, W-1-j)
    float4 x[4];
#pragma unroll
    for (int z = 0; z < 4; ++z) x[z] = *reinterpret_cast<const float4*>(Q + z * plane + o);
    const float ee[4] = {x[0].x, x[0].y, x[0].z, x[0].w}, oe[4] = {x[1].x, x[1].y, x[1].z, x[1].w};
    const float eo[4] = {x[2].x, x[2].y, x[2].z, x[2].w}, oo[4] = {x[3].x, x[3].y, x[3].z, x[3].w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float p = ee[e] + oe[e], m = ee[e] - oe[e], u = eo[e] + oo[e], v = eo[e] - oo[e];
        a[e] = p + u;
        b[e] = m + v;
        c[e] = p - u;
        d[e] = m - v;
    }
    float* up = Z + (size_t)i * ldz;
    float* dn = Z + (size_t)(H - 1 - i) * ldz;
    const bool two = 2 * i != H - 1;
    if (vec && j0 + 3 < hW) {
        *reinterpret_cast<float4*>(up + j0) = make_float4(a[0], a[1], a[2], a[3]);
        *reinterpret_cast<float4*>(up + W - 4 - j0) = make_float4(c[3], c[2], c[1], c[0]);
        if (two) {
            *reinterpret_cast<float4*>(dn + j0) = make_float4(b[0], b[1], b[2], b[3]);
            *reinterpret_cast<float4*>(dn + W - 4 - j0) = make_float4(d[3], d[2], d[1], d[0]);
        }
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (j0 + e >= hW) continue;
            up[j0 + e] = a[e];
            if (two) dn[j0 + e] = b[e];
            if (2 * (j0 + e) == W - 1) continue;
            up[W - 1 - j0 - e] = c[e];
            if (two) dn[W - 1 - j0 - e] = d[e];
        }
    }
}

// The basis halves of a side of N, one per parity s of the frequency k = 2a + s, over positions
// i < he = ceil(N / 2): position-major (Q: [i][a], stages 1 and 2) and frequency-major (F: [a][i],
// stages 3 and 4), zero in the pitch padding and for k = N of an odd side.  The argument is
// reduced exactly in integers before the FP64 cospi.
__global__ void k_build_halves(float* F0, float* F1, float* Q0, float* Q1, int N, int he, int ld) {
    const size_t total = (size_t)he * ld;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
         t += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / ld), a = (int)(t % ld);
        if (a >= he) {
            F0[t] = F1[t] = Q0[t] = Q1[t] = 0.f;
            continue;
        }
        for (int s = 0; s < 2; ++s) {
            const int k = 2 * a + s;
            double v = 0.0;
            if (k < N) {
                const long long m = ((long long)(2 * i + 1) * k) % (4LL * N);
                v = (k == 0 ? sqrt(1.0 / N) : sqrt(2.0 / N)) * cospi((double)m / (2.0 * N));
            }
            (s ? F1 : F0)[(size_t)a * ld + i] = (float)v;
            (s ? Q1 : Q0)[t] = (float)v;
        }
    }
}

// Eigenvalues l_k = 2 - 2 cos(pi k / N) = 4 sin^2(pi k / 2N) of S^T S (Sec. 3.3), zero-padded.
__global__ void k_build_lambda(float* lam, int N, int Np) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < Np; k += gridDim.x * blockDim.x) {
        double v = 0.0;
        if (k < N) {
            const double s = sinpi((double)k / (2.0 * N));
            v = 4.0 * s * s;
        }
        lam[k] = (float)v;
    }
}

inline int rup(int x, int m) { return (x + m - 1) / m * m; }
inline int half_up(int n) { return (n + 1) / 2; }
inline int half_ld(int n) { return rup(half_up(n), 4); }
// floats of one side's basis halves
inline size_t halves_floats(int n) { return (size_t)4 * half_up(n) * half_ld(n); }

struct Halves {
    const float *F0, *F1, *Q0, *Q1;
    int ld;
};
Halves halves(const float* mem, int n) {
    const size_t p = (size_t)half_up(n) * half_ld(n);
    return {mem, mem + p, mem + 2 * p, mem + 3 * p, half_ld(n)};
}
void build_halves(float* mem, int n, cudaStream_t s) {
    const Halves h = halves(mem, n);
    const size_t p = (size_t)half_up(n) * h.ld;
    const int blocks = (int)std::min<size_t>((p + 255) / 256, 2048);
    k_build_halves<<<blocks, 256, 0, s>>>(mem, mem + p, mem + 2 * p, mem + 3 * p, n, half_up(n),
                                          h.ld);
}

template <class C>
dim3 quad_grid(int M, int N) {
    return dim3((N + C::BN - 1) / C::BN, (M + C::BM - 1) / C::BM, 4);
}

// The medium tile's ring is the default limit of 48 KB, with the spectrum's reduction above it.
// Set once per plan; the scratch form's sides (at most 256) take the small tile.
cudaError_t quad_attributes() {
    return cudaFuncSetAttribute(k_quad_gemm_f32<TileM, true>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, TileM::SMEM);
}
static_assert(TileL::SMEM < 47 * 1024 && TileS::SMEM < 47 * 1024 && TileM::SMEM <= 48 * 1024, "");

template <class C, bool SPECTRUM>
cudaError_t quad_launch(const QuadArgs& f, cudaStream_t s) {
    return launch_kernel(f.pdl != 0, k_quad_gemm_f32<C, SPECTRUM>, quad_grid<C>(f.M, f.N), C::T, C::SMEM,
                         s, f);
}

// Tile of a launch (0 large, 1 medium, 2 small): the least busy-SM time, in large tiles.  A
// block's multiply-adds take their share of an SM whether or not another block runs beside it, so
// a launch lasts as long as the SM with the most blocks; a medium tile is a quarter and a small
// one a sixteenth of the large tile's work at 0.88 and 0.62 of its rate.  Measured (us per
// application, large / medium / small): 512^2 139 / 68 / 55, 701 x 1003 204 / 131 / 114, 1024^2
// 234 / 148 / 160, 1500^2 324 / 349 / 434, 2000 x 1100 553 / 365 / 452, 4096^2 4540 / 5153 / 6711.
int quad_tile(int M, int N) {
    constexpr unsigned kSms = 152;
    auto waves = [](dim3 g) { return (double)((g.x * g.y * g.z + kSms - 1) / kSms); };
    const double l = waves(quad_grid<TileL>(M, N));
    const double m = waves(quad_grid<TileM>(M, N)) / 4 / 0.88;
    const double t = waves(quad_grid<TileS>(M, N)) / 16 / 0.62;
    return l <= m && l <= t ? 0 : m <= t ? 1 : 2;
}

template <bool SPECTRUM>
cudaError_t quad_stage(const QuadArgs& f, cudaStream_t s) {
    switch (quad_tile(f.M, f.N)) {
        case 0: return quad_launch<TileL, SPECTRUM>(f, s);
        case 1: return quad_launch<TileM, SPECTRUM>(f, s);
        default: return quad_launch<TileS, SPECTRUM>(f, s);
    }
}

dim3 fold_grid(int hH, int hW) { return dim3((hW + 255) / 256, (hH + 3) / 4); }

// Floats of the two intermediates of fold_products.
size_t quad_floats(int H, int W) {
    return 4 * std::max((size_t)half_up(H) * half_ld(W), (size_t)half_up(W) * half_ld(H));
}

// The map from the plane R (pitch ldr) into Z (pitch ldz), with the two sides' basis halves,
// eigenvalues and two intermediates of quad_floats(H, W) floats.  `base` carries the state,
// scratch and flags.
cudaError_t fold_products(const float* R, int ldr, float* Z, int ldz, int H, int W, float tau,
                          const Halves& hn, const Halves& hm, const float* lamN,
                          const float* lamM, float* T1, float* T2, const QuadArgs& base,
                          cudaStream_t s) {
    const int hH = half_up(H), hW = half_up(W), ph = half_ld(H), pw = half_ld(W);
    const size_t rows = (size_t)hH * pw, cols = (size_t)hW * ph;   // quadrant planes
    auto aligned = [&](const float* p, int ld) {
        return W % 4 == 0 && ld % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0;
    };
    const bool pdl = base.pdl != 0;
    cudaError_t e = launch_kernel(pdl, k_quad_fold, fold_grid(hH, hW), dim3(64, 4), 0, s, R, ldr, H, W,
                                  T1, pw, (int)aligned(R, ldr), base.st, base.skip_if_done);
    if (e != cudaSuccess) return e;
    QuadArgs f = base;
    f.A = T1; f.sa = rows; f.lda = pw; f.B0 = hn.Q0; f.B1 = hn.Q1; f.ldb = ph; f.by_q = 0;
    f.C = T2; f.sc = cols; f.ldc = ph; f.M = hW; f.N = hH; f.K = hH;
    if ((e = quad_stage<false>(f, s)) != cudaSuccess) return e;
    f.A = T2; f.sa = cols; f.lda = ph; f.B0 = hm.Q0; f.B1 = hm.Q1; f.ldb = pw; f.by_q = 1;
    f.C = T1; f.sc = rows; f.ldc = pw; f.M = hH; f.N = hW; f.K = hW;
    f.n_k = H; f.n_l = W; f.lam_k = lamN; f.lam_l = lamM; f.scale = tau;
    if ((e = quad_stage<true>(f, s)) != cudaSuccess) return e;
    f.A = T1; f.sa = rows; f.lda = pw; f.B0 = hn.F0; f.B1 = hn.F1; f.ldb = ph; f.by_q = 0;
    f.C = T2; f.sc = cols; f.ldc = ph; f.M = hW; f.N = hH; f.K = hH;
    if ((e = quad_stage<false>(f, s)) != cudaSuccess) return e;
    f.A = T2; f.sa = cols; f.lda = ph; f.B0 = hm.F0; f.B1 = hm.F1; f.ldb = pw; f.by_q = 1;
    f.C = T1; f.sc = rows; f.ldc = pw; f.M = hH; f.N = hW; f.K = hW;
    if ((e = quad_stage<false>(f, s)) != cudaSuccess) return e;
    return launch_kernel(pdl, k_quad_unfold, fold_grid(hH, hW), dim3(64, 4), 0, s, T1, pw, H, W, Z, ldz,
                         (int)aligned(Z, ldz), base.st, base.skip_if_done);
}

// ---- full-size products, for taped solves and their adjoint -----------------------------------
// The gradient divides by W = sqrt(C^2 V^2 + delta^2) of edges whose V is close to zero, so it
// carries the rounding of the solves times up to 1 / delta: 1e-7 of z_U, where the quadrant
// products round otherwise than the full ones, moves dL/dX by 1e-4 (both as far from the float64
// gradient; with the full-size products two versions of the library agree to 2e-7).  So that
// gradients do not move, the solves that a tape records and the adjoint's keep the full-size
// products and their order of summation: T1 = R P_M, T2 = (T1^T P_N) scaled, T1 = T2 P_N^T,
// Z = T1 P_M^T, each output one chain of multiply-adds along k.  128 x 128 tiles, 8 x 8 a thread,
// operands staged through registers: 43 TFLOP/s at 4096^2, of twice the quadrants' work.  A
// recorded solve with its adjoint at 486 x 931, four steps, takes 595 ms (679 before the stencils'
// one-wave rows and the dependent launches).
constexpr int kFullTile = 128;

enum Epi : int { EPI_TRANS = 0, EPI_EIG = 1, EPI_ZU_RHO = 2 };

struct EpiArgs {
    float* C;          // output
    int ldc;
    int vm, vn;        // valid extents (EPI_EIG: W, H; EPI_ZU_RHO: H, W)
    const float* lam_m;
    const float* lam_n;
    float scale;       // tau (EPI_EIG)
    const float* rU;   // EPI_ZU_RHO: residual plane, pitch ldc
    DevState* st;
    double* partials;
    int flexible;
};

// C[m][n] = sum_k A[m][k] B[n][k], M and N multiples of 128; A rows >= a_rows and k >= K read 0.
template <int EPI>
__global__ void __launch_bounds__(256)
k_gemm_tn_f32(const float* __restrict__ A, int lda, int a_rows, const float* __restrict__ B,
              int ldb, int K, EpiArgs ep, int skip_if_done) {
    if (skip_if_done && ep.st != nullptr && ep.st->done) return;
    constexpr int BM = kFullTile, BN = kFullTile, BK = 8;
    __shared__ __align__(16) float As[2][BK][BM + 4];
    __shared__ __align__(16) float Bs[2][BK][BN + 4];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    // loader mapping: 128 rows x 8 k per operand; thread -> (row, 4 consecutive k)
    const int lr = tid >> 1, lk = (tid & 1) * 4;
    const bool arow = (m0 + lr) < a_rows;
    const float* Ap = A + (size_t)(m0 + lr) * lda;
    const float* Bp = B + (size_t)(n0 + lr) * ldb;

    auto load4 = [&](const float* p, bool rowok, int k, float (&r)[4]) {
        if (rowok && k + 3 < K) {
            float4 v = *reinterpret_cast<const float4*>(p + k);
            r[0] = v.x; r[1] = v.y; r[2] = v.z; r[3] = v.w;
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) r[c] = (rowok && k + c < K) ? p[k + c] : 0.f;
        }
    };

    float ra[4], rb[4];
    load4(Ap, arow, lk, ra);
    load4(Bp, true, lk, rb);
#pragma unroll
    for (int c = 0; c < 4; ++c) { As[0][lk + c][lr] = ra[c]; Bs[0][lk + c][lr] = rb[c]; }
    __syncthreads();

    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;

    const int nk = (K + BK - 1) / BK;
    for (int kt = 0; kt < nk; ++kt) {
        const int buf = kt & 1;
        if (kt + 1 < nk) {
            load4(Ap, arow, (kt + 1) * BK + lk, ra);
            load4(Bp, true, (kt + 1) * BK + lk, rb);
        }
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][64 + ty * 4]);
            const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * 4]);
            const float4 b1 = *reinterpret_cast<const float4*>(&Bs[buf][kk][64 + tx * 4]);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        if (kt + 1 < nk) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                As[buf ^ 1][lk + c][lr] = ra[c];
                Bs[buf ^ 1][lk + c][lr] = rb[c];
            }
        }
        __syncthreads();
    }

    CSum part;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int m = m0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + (i - 4));
        float row = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int n = n0 + (j < 4 ? tx * 4 + j : 64 + tx * 4 + (j - 4));
            const float v = acc[i][j];
            if constexpr (EPI == EPI_TRANS) {
                ep.C[(size_t)n * ep.ldc + m] = v;
            } else if constexpr (EPI == EPI_EIG) {
                float o = 0.f;
                if (m < ep.vm && n < ep.vn && (m | n) != 0) o = ep.scale * v / (ep.lam_m[m] + ep.lam_n[n]);
                ep.C[(size_t)m * ep.ldc + n] = o;
            } else {
                if (m < ep.vm && n < ep.vn) {
                    ep.C[(size_t)m * ep.ldc + n] = v;
                    row += ep.rU[(size_t)m * ep.ldc + n] * v;
                }
            }
        }
        if constexpr (EPI == EPI_ZU_RHO) part.add(row);
    }
    if constexpr (EPI == EPI_ZU_RHO) {
        double vv[1] = {part.value()}, tot[1];
        const Blk blk = single_blk();
        if (grid_reduce<1>(vv, ep.partials, &ep.st->counter, tot, blk.nblk, blk.bid) && tid == 0)
            finish_rho(ep.st, tot[0], ep.flexible);
    }
}

// P[i][k] = c_k cos(pi k (2i+1) / (2N)) and its transpose, zero-padded to Np x Np.  The
// argument is reduced exactly in integers before the FP64 cospi.
__global__ void k_build_full(float* P, float* PT, int N, int Np) {
    const size_t total = (size_t)Np * Np;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
         t += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / Np), k = (int)(t % Np);
        double v = 0.0;
        if (i < N && k < N) {
            const long long m = ((long long)(2 * i + 1) * k) % (4LL * N);
            const double ck = k == 0 ? sqrt(1.0 / N) : sqrt(2.0 / N);
            v = ck * cospi((double)m / (2.0 * N));
        }
        P[(size_t)i * Np + k] = (float)v;
        PT[(size_t)k * Np + i] = (float)v;
    }
}

template <int EPI>
cudaError_t full_gemm(const float* A, int lda, int a_rows, const float* B, int ldb, int M, int N,
                      int K, const EpiArgs& ep, int skip, cudaStream_t s) {
    dim3 grid(N / kFullTile, M / kFullTile);
    k_gemm_tn_f32<EPI><<<grid, 256, 0, s>>>(A, lda, a_rows, B, ldb, K, ep, skip);
    return cudaGetLastError();
}

// (always with rho: only CG runs take these products)
cudaError_t full_products(const DctPlan& d, const float* rU, float* zU, int ld, DevState* st,
                          int flexible, double* partials, int skip, cudaStream_t s) {
    const int H = d.H, W = d.W, Hp = d.Hp, Wp = d.Wp;
    cudaError_t e;
    EpiArgs ep{};
    ep.st = st;
    ep.partials = partials;
    ep.flexible = flexible;
    // stage 1: T1[l][i] = sum_j R[i][j] PMT[l][j]
    ep.C = d.T1; ep.ldc = Hp;
    e = full_gemm<EPI_TRANS>(rU, ld, H, d.PMT, Wp, Hp, Wp, W, ep, skip, s);
    if (e != cudaSuccess) return e;
    // stage 2: T2[l][k] = tau sum_i T1[l][i] PNT[k][i] / (m_l + l_k), (0,0) -> 0
    ep.C = d.T2; ep.ldc = Hp; ep.vm = W; ep.vn = H; ep.lam_m = d.lamM; ep.lam_n = d.lamN;
    ep.scale = d.tau;
    e = full_gemm<EPI_EIG>(d.T1, Hp, Wp, d.PNT, Hp, Wp, Hp, H, ep, skip, s);
    if (e != cudaSuccess) return e;
    // stage 3: T1[i][l] = sum_k T2[l][k] PN[i][k]
    ep.C = d.T1; ep.ldc = Wp;
    e = full_gemm<EPI_TRANS>(d.T2, Hp, Wp, d.PN, Hp, Wp, Hp, H, ep, skip, s);
    if (e != cudaSuccess) return e;
    // stage 4: Z[i][j] = sum_l T1[i][l] PM[j][l]
    ep.C = zU; ep.ldc = ld; ep.vm = H; ep.vn = W; ep.rU = rU;
    return full_gemm<EPI_ZU_RHO>(d.T1, Wp, Hp, d.PM, Wp, Hp, Wp, W, ep, skip, s);
}

}  // namespace

// blocks of the grid-reduced second product in its smallest tile
int dct_max_blocks(int H, int W) {
    const dim3 g = quad_grid<TileS>(half_up(H), half_up(W));
    return (int)(g.x * g.y * g.z);
}

size_t dct_bytes(int H, int W, int prec) {
    const size_t Hp = rup(H, 128), Wp = rup(W, 128);
    size_t n = halves_floats(H) + Hp + Wp + 2 * Hp * Wp;
    if (H != W) n += halves_floats(W);
    size_t bytes = n * sizeof(float) + 4096;
    if (prec != IRLS_PREC_FP32) bytes += umma_dct_bytes(H, W, prec);
    return bytes + fft_dct_bytes(H, W);   // the fast-transform tables at the tail
}

cudaError_t dct_setup(DctPlan& d, int H, int W, int prec, float tau, char* mem) {
    d.H = H; d.W = W; d.Hp = rup(H, 128); d.Wp = rup(W, 128); d.prec = prec; d.tau = tau;
    const size_t Hp = d.Hp, Wp = d.Wp;
    float* f = reinterpret_cast<float*>(mem);
    d.T1 = f; f += Hp * Wp;
    d.T2 = f; f += Hp * Wp;
    d.lamN = f; f += Hp;
    d.lamM = (H != W) ? f : d.lamN;
    f += Wp;
    d.halvesN = f; f += halves_floats(H);
    d.halvesM = (H != W) ? f : d.halvesN;
    build_halves(d.halvesN, H, 0);
    if (H != W) build_halves(d.halvesM, W, 0);
    cudaError_t e = quad_attributes();
    if (e != cudaSuccess) return e;
    k_build_lambda<<<8, 256>>>(d.lamN, H, d.Hp);
    if (H != W) k_build_lambda<<<8, 256>>>(d.lamM, W, d.Wp);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    d.umma_ok = 0;
    d.fft = 0;
    {
        char* mt = mem + (dct_bytes(H, W, prec) - fft_dct_bytes(H, W));
        mt = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(mt) + 255) & ~uintptr_t(255));
        if ((e = fft_dct_setup(d, mt)) != cudaSuccess) return e;
    }
    if (prec != IRLS_PREC_FP32) {
        char* m16 = mem + (dct_bytes(H, W, IRLS_PREC_FP32) - fft_dct_bytes(H, W) - 4096);
        m16 = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(m16) + 1023) & ~uintptr_t(1023));
        e = umma_dct_setup(d, m16);
    }
    return e;
}

void dct_release(DctPlan& d) {
    if (d.full_mem) cudaFree(d.full_mem);
    d.full_mem = nullptr;
    umma_dct_release(d);
}

// The full-size bases of the float32 dense form, on the first solve of a plan that needs them
// (kept with the plan).  Nothing for the other forms.
cudaError_t dct_full_setup(DctPlan& d, cudaStream_t s) {
    if (d.full_mem || !dct_runs_full(d)) return cudaSuccess;
    const size_t n = (size_t)d.Hp * d.Hp, m = d.H != d.W ? (size_t)d.Wp * d.Wp : 0;
    void* mem = nullptr;
    cudaError_t e = cudaMalloc(&mem, 2 * (n + m) * sizeof(float));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e;
    }
    d.PN = static_cast<float*>(mem);
    d.PNT = d.PN + n;
    d.PM = m ? d.PNT + n : d.PN;
    d.PMT = m ? d.PM + m : d.PNT;
    k_build_full<<<1024, 256, 0, s>>>(d.PN, d.PNT, d.H, d.Hp);
    if (m) k_build_full<<<1024, 256, 0, s>>>(d.PM, d.PMT, d.W, d.Wp);
    if ((e = cudaGetLastError()) != cudaSuccess) {
        cudaFree(mem);
        return e;
    }
    d.full_mem = mem;   // (set last: a plan that has it has the bases)
    return cudaSuccess;
}
cudaError_t dct_reset(const DctPlan& d, cudaStream_t s) { return umma_dct_reset(d, s); }
bool dct_stall(DctPlan& d, int on) { return umma_dct_stall(d, on); }

cudaError_t dct_apply(const DctPlan& d, const float* rU, float* zU, int ld, DevState* st,
                      int reduce_rho, const StencilArgs& a, double* partials, int skip_if_done,
                      cudaStream_t s, const float* src, int ld_src) {
    if (d.fft) return fft_dct_apply(d, rU, zU, ld, st, reduce_rho, a, partials, skip_if_done, s);
    if (d.prec != IRLS_PREC_FP32)
        return umma_dct_apply(d, rU, zU, ld, st, reduce_rho, a, partials, skip_if_done, s, src,
                              ld_src);
    if (a.full) return full_products(d, rU, zU, ld, st, a.flexible, partials, skip_if_done, s);
    QuadArgs base{};
    base.st = st;
    base.partials = partials;
    base.rho = reduce_rho;
    base.flexible = a.flexible;
    base.skip_if_done = skip_if_done;
    base.pdl = a.pdl;
    return fold_products(rU, ld, zU, ld, d.H, d.W, d.tau, halves(d.halvesN, d.H),
                         halves(d.halvesM, d.W), d.lamN, d.lamM, d.T1, d.T2, base, s);
}

// Floats of scratch that dct_apply_fp32_scratch needs for an H x W image.
size_t dct_scratch_floats(int H, int W) {
    size_t n = halves_floats(H) + rup(H, 4) + 2 * quad_floats(H, W);
    if (H != W) n += halves_floats(W) + rup(W, 4);
    return n;
}

// The float32 Laplacian preconditioner on caller-provided scratch: builds the basis halves into
// `work` and runs the four products from R into Z (pitch W both).  Every scratch element that is
// read is written earlier in the same call.
cudaError_t dct_apply_fp32_scratch(const float* R, float* Z, int H, int W, float tau, float* work,
                                   cudaStream_t s) {
    float* f = work;
    float* bn = f; f += halves_floats(H);
    float* bm = bn;
    if (H != W) { bm = f; f += halves_floats(W); }
    float* lamN = f; f += rup(H, 4);
    float* lamM = lamN;
    if (H != W) { lamM = f; f += rup(W, 4); }
    float* T1 = f; f += quad_floats(H, W);
    float* T2 = f;
    build_halves(bn, H, s);
    if (H != W) build_halves(bm, W, s);
    k_build_lambda<<<2, 256, 0, s>>>(lamN, H, H);
    if (H != W) k_build_lambda<<<2, 256, 0, s>>>(lamM, W, W);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    QuadArgs base{};
    base.pdl = 1;
    return fold_products(R, W, Z, W, H, W, tau, halves(bn, H), halves(bm, W), lamN, lamM, T1, T2,
                         base, s);
}

}  // namespace irls
