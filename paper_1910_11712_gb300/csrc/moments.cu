// Kernel (d): contour moments and the block Hankel matrices, FP64.
//
// By Keldysh's theorem (Sec. 2 Eq. (resolvent)) the quadrature of zeta^k T(z)^{-1} V over
// Gamma keeps only the eigenvalues inside Gamma. With the trapezoid nodes/weights:
//   S_k = sum_j w_j zeta_j^k Y_j  (Y_j = T(z_j)^{-1} V),    mu_k = V^H S_k,    k < 2M,
//   H = [mu_{a+b}],  H< = [mu_{a+b+1}]  (a, b < M; LM x LM, column-major).
// moments_df_kernel (complex64 factors, Y in double-float pairs): one thread per entry (i, l) of the n x L block reads
// Y_j(i, l) once for every point j (ascending) and keeps the K = 2M accumulators in registers; the coefficients
// c_jk = w_j zeta_j^k sit in shared memory. Bound by FP32 issue.
// moments_oz_kernel (FP64, up to 192 points): exact digit products on the tensor core, below.
// moments_kernel and moments_kernel_generic (more points): as the first, in FP64 (1.75 FMA/clk/SM on this part, so with
// 2M*4 FMAs per 16 bytes read bound by FP64 issue, not by HBM).
// mu_k = V^H S_k is a product of gemm.cu, split over the rows with a fixed-order reduction (no
// atomics), so results do not depend on scheduling.
#include <algorithm>

#include "df_arith.cuh"
#include "nep_common.cuh"
#include "oz.cuh"

namespace nep {

template <int K>
__global__ void __launch_bounds__(256) moments_kernel(int64_t nl, int N, const zd* __restrict__ coef,
                                                      const zd* __restrict__ Y, zd* __restrict__ S) {
    extern __shared__ zd cs[];  // N x K
    for (int t = threadIdx.x; t < N * K; t += blockDim.x) cs[t] = coef[(t / K) + (int64_t)N * (t % K)];
    __syncthreads();
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nl) return;
    zd acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = mk(0.0, 0.0);
    for (int j = 0; j < N; ++j) {
        const zd y = Y[(int64_t)j * nl + e];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = fma_(acc[k], cs[j * K + k], y);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) S[(int64_t)k * nl + e] = acc[k];
}

// generic K (loop over k in chunks of 8 accumulators)
__global__ void __launch_bounds__(256) moments_kernel_generic(int64_t nl, int N, int K, const zd* __restrict__ coef,
                                                              const zd* __restrict__ Y, zd* __restrict__ S) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nl) return;
    for (int k0 = 0; k0 < K; k0 += 8) {
        zd acc[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] = mk(0.0, 0.0);
        for (int j = 0; j < N; ++j) {
            const zd y = Y[(int64_t)j * nl + e];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k0 + k < K) acc[k] = fma_(acc[k], coef[j + (int64_t)N * (k0 + k)], y);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k0 + k < K) S[(int64_t)(k0 + k) * nl + e] = acc[k];
    }
}

// ------------------------------------------------------------------ FP64 moments on the tensor core
// The moments are a contraction, K x N coefficients by N x (n L) values, done with exact digit products (oz.cuh).
// A warp takes 8 columns: its B fragments come straight from global memory (lane: column lane / 4,
// nodes lane % 4 and + 4 of each 8; the column's exponent from a first pass over it, the digits from a
// second that hits L1), the coefficients' digits are built once per CTA in the fragments' order in shared
// memory. Columns with a non-finite entry or an extreme exponent take FP64 sums as moments_kernel does, and so does
// every result that the guard (oz.cuh) finds too small for the digits.
// n L = 524288, N = 64, K = 16: 0.486 ms (FP64 FMAs: 3.56, at the FP64 pipe's rate; HBM alone: 0.10). Error
// against a 113-bit sum: 4.7e-17 (N <= 64) and 8.3e-17 (N = 192) of the result's norm, FP64 FMAs 2.7e-16 to
// 6.7e-16. On an ellipse the guard takes part: 0.534 ms. What bounds it: latency with 16 warps an SM (128 registers); the
// MMA pipe of mma.sync is the busiest unit, 54 % (issue 42 %, DRAM 17 %).
namespace oz {
constexpr int KC = CH / 8;        // 16-wide MMA steps per chunk (8 nodes)
constexpr int FRAG = 32 * 4;      // words of one A fragment
}  // namespace oz

// MT: tiles of 8 moments (1 or 2) of this CTA's share (blockIdx.y); nch chunks of CH nodes
template <int MT>
__global__ void __launch_bounds__(256, 2)
    moments_oz_kernel(int64_t nl, int N, int K, int nch, const zd* __restrict__ coef, const zd* __restrict__ Y,
                      zd* __restrict__ Sout) {
    using namespace oz;
    extern __shared__ uint4 afrag[];  // [chunk][MT][KC][S][32 lanes], then the guard's [chunk][KC][32 lanes]
    __shared__ int ea[8 * MT], bad, guarded;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int kbase = blockIdx.y * 8 * MT;
    auto cval = [&](int j, int k) { return j < N && k < K ? coef[j + (int64_t)N * k] : mk(0.0, 0.0); };
    if (tid == 0) bad = guarded = 0;
    if (tid < 8 * MT) ea[tid] = 0;
    __syncthreads();
    for (int e = tid; e < N * 8 * MT; e += blockDim.x) {
        const int k = e / N, j = e - k * N;
        const zd c = cval(j, kbase + k);
        atomicMax(&ea[k], exp_field(c));
    }
    __syncthreads();
    if (tid < 8 * MT) {
        if (ea[tid] != 0 && (ea[tid] < EXP_LO || ea[tid] > EXP_HI)) bad = 1;
        if (ea[tid] == 0) ea[tid] = E_ZERO;
    }
    __syncthreads();
    const bool slow_all = bad != 0;
    if (!slow_all) {
        // word w of lane l of the fragment: row l / 4 (+ 8: the Im row) for w odd, node l % 4 (+ 4 for w >= 2)
        for (int e = tid; e < nch * MT * KC * 32 * 4; e += blockDim.x) {
            const int w = e & 3, l = (e >> 2) & 31, kc = (e >> 7) % KC, mt = (e >> 7) / KC % MT, ch = (e >> 7) / (KC * MT);
            const int k = 8 * mt + l / 4, j = ch * CH + kc * 8 + (l & 3) + ((w & 2) ? 4 : 0);
            const zd c = cval(j, kbase + k);
            const int E = ea[k];
            const unsigned long long p = fixed62((w & 1) ? c.im : c.re, E), q = fixed62((w & 1) ? c.re : -c.im, E);
            unsigned* f = reinterpret_cast<unsigned*>(afrag) + (((size_t)(ch * MT + mt) * KC + kc) * S) * FRAG + l * 4 + w;
#pragma unroll
            for (int t = 0; t < S; ++t) f[t * FRAG] = digits2(p, q, S - 1 - t);  // the highest digit first
        }
        // the guard's leading bits: rows 0 .. 7 the first tile of 8 moments, rows 8 .. 15 the second. With every
        // coefficient at least 2/64 of its row's scale it is met, since a column's largest entry has 32/64 of its own
        for (int e = tid; e < nch * KC * 32 * 4; e += blockDim.x) {
            const int w = e & 3, l = (e >> 2) & 31, kc = (e >> 7) % KC, ch = (e >> 7) / KC;
            const int k = l / 4 + ((w & 1) ? 8 : 0), j = ch * CH + kc * 8 + (l & 3) + ((w & 2) ? 4 : 0);
            const unsigned f = k < 8 * MT ? lead(cval(j, kbase + k), ea[k]) : 0u;
            reinterpret_cast<unsigned*>(afrag + (size_t)nch * MT * KC * S * 32)[e] = lead2(f);
            if (f < 2 && k < 8 * MT && j < N && ea[k] != E_ZERO) guarded = 1;
        }
    }
    __syncthreads();
    const bool guard = guarded != 0;
    const int64_t tiles = (nl + 7) / 8;
    for (int64_t tile = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp; tile < tiles;
         tile += (int64_t)gridDim.x * (blockDim.x >> 5)) {
        const int64_t e0 = tile * 8, col = e0 + (lane >> 2);
        const int jl = lane & 3;
        const zd* yc = Y + col;
        const bool in = col < nl;
        int E = 0;
#pragma unroll 4
        for (int j = jl; j < N; j += 4) {
            if (in) E = max(E, exp_field(yc[(int64_t)j * nl]));
        }
        E = max(E, __shfl_xor_sync(0xffffffffu, E, 1));
        E = max(E, __shfl_xor_sync(0xffffffffu, E, 2));
        const bool okc = E == 0 || (E >= EXP_LO && E <= EXP_HI);
        if (slow_all || __any_sync(0xffffffffu, !okc)) {
            for (int o = lane; o < 64 * MT; o += 32) {
                const int64_t c = e0 + (o & 7);
                const int k = kbase + (o >> 3);
                if (c >= nl || k >= K) continue;
                zd acc = mk(0.0, 0.0);
                for (int j = 0; j < N; ++j) acc = fma_(acc, coef[j + (int64_t)N * k], Y[(int64_t)j * nl + c]);
                Sout[(int64_t)k * nl + c] = acc;
            }
            continue;
        }
        if (E == 0) E = E_ZERO;
        double out[MT][4];
        float G[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // the guard of both tiles over all nodes
        for (int ch = 0; ch < nch; ++ch) {
            float D[MT][S][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int t = 0; t < S; ++t)
#pragma unroll
                    for (int q = 0; q < 4; ++q) D[m][t][q] = 0.0f;
            const int kcs = min(KC, (N - ch * CH + 7) / 8);
            const uint4* af = afrag + (size_t)ch * MT * KC * S * 32 + lane;
            const uint4* gf = afrag + (size_t)nch * MT * KC * S * 32 + lane;
#pragma unroll 1
            for (int kc = 0; kc < kcs; ++kc) {
                const int j = ch * CH + kc * 8 + jl;
                const zd y0 = in && j < N ? yc[(int64_t)j * nl] : mk(0.0, 0.0);
                const zd y1 = in && j + 4 < N ? yc[(int64_t)(j + 4) * nl] : mk(0.0, 0.0);
                if (guard) mma16816(G, gf[(size_t)(ch * KC + kc) * 32], lead2(lead(y0, E)), lead2(lead(y1, E)));
                const unsigned long long r0 = fixed62(y0.re, E), i0 = fixed62(y0.im, E);
                const unsigned long long r1 = fixed62(y1.re, E), i1 = fixed62(y1.im, E);
                unsigned b0[S], b1[S];
#pragma unroll
                for (int t = 0; t < S; ++t) {
                    b0[t] = digits2(r0, i0, S - 1 - t);
                    b1[t] = digits2(r1, i1, S - 1 - t);
                }
#pragma unroll
                for (int ta = 0; ta < S; ++ta)
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        const uint4 a = af[(size_t)((m * KC + kc) * S + ta) * 32];
#pragma unroll
                        for (int tb = 0; ta + tb < S; ++tb) mma16816(D[m][ta + tb], a, b0[tb], b1[tb]);
                    }
            }
            // columns 2 (lane % 4) + (q & 1); rows lane / 4 (Re for q < 2, else Im)
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int Eb = __shfl_sync(0xffffffffu, E, 4 * (2 * (lane & 3) + (q & 1)));
                    const double sv = combine(D[m], q, ea[8 * m + (lane >> 2)], Eb);
                    out[m][q] = ch == 0 ? sv : out[m][q] + sv;
                }
        }
        if (guard) {
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int Eb = __shfl_sync(0xffffffffu, E, 4 * (2 * (lane & 3) + q));
                    const bool weak = G[2 * m + q] < GUARD && ea[8 * m + (lane >> 2)] != E_ZERO && Eb != E_ZERO;
                    const unsigned todo = __ballot_sync(0xffffffffu, weak);
                    if (todo) {
                        const zd s = fp64_sums(todo, N, coef + (int64_t)N * (kbase + 8 * m), N, 1, false,
                                               Y + e0 + q, 2, nl);
                        if (weak) out[m][q] = s.re, out[m][2 + q] = s.im;
                    }
                }
        }
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const int k = kbase + 8 * m + (lane >> 2);
            const int64_t c = e0 + 2 * (lane & 3);
            if (k < K) {
                if (c < nl) Sout[(int64_t)k * nl + c] = mk(out[m][0], out[m][2]);
                if (c + 1 < nl) Sout[(int64_t)k * nl + c + 1] = mk(out[m][1], out[m][3]);
            }
        }
    }
}

// The digits of up to 192 nodes' coefficients fit in shared memory
template <int MT>
static int launch_moments_oz(int64_t nl, int N, int K, const zd* coef, const zd* Y, zd* S, cudaStream_t st) {
    const int nch = ceil_div(N, oz::CH);
    const size_t sm = (size_t)nch * oz::KC * (MT * oz::S + 1) * oz::FRAG * 4;
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 152;
    }();
    NEP_CUDA(allow_max_dynamic_smem(moments_oz_kernel<MT>));
    const int gy = ceil_div(K, 8 * MT), per = sm <= 112 * 1024 ? 2 : 1;
    const int gx = (int)std::min<int64_t>((nl + 63) / 64, std::max(1, per * sms / gy));
    moments_oz_kernel<MT><<<dim3(gx, gy), 256, sm, st>>>(nl, N, K, nch, coef, Y, S);
    NEP_CHECK_LAUNCH();
    return NEP_OK;
}

int launch_moments(int n, int L, int N, int K, const zd* coef, const zd* Y, zd* S, cudaStream_t st) {
    const int64_t nl = (int64_t)n * L;
    const int blocks = ceil_div(nl, 256);
    const size_t sm = sizeof(zd) * (size_t)N * K;
    if (nl >= 1 && N <= 3 * oz::CH && K >= 1)
        return K <= 8 ? launch_moments_oz<1>(nl, N, K, coef, Y, S, st) : launch_moments_oz<2>(nl, N, K, coef, Y, S, st);
    if (K == 16 && sm <= 96 * 1024) {
        NEP_CUDA(allow_max_dynamic_smem(moments_kernel<16>));
        moments_kernel<16><<<blocks, 256, sm, st>>>(nl, N, coef, Y, S);
    } else if (K == 8 && sm <= 96 * 1024) {
        NEP_CUDA(allow_max_dynamic_smem(moments_kernel<8>));
        moments_kernel<8><<<blocks, 256, sm, st>>>(nl, N, coef, Y, S);
    } else {
        moments_kernel_generic<<<blocks, 256, 0, st>>>(nl, N, K, coef, Y, S);
    }
    NEP_CHECK_LAUNCH();
    return NEP_OK;
}

// The moments from Y held as double-float pairs (complex64 factors, the refinement's form): the
// accumulation in double-float arithmetic (coefficients split once per CTA), S written in FP64,
// and each Y element returned to FP64 in place after it is read.
template <int K>
__global__ void __launch_bounds__(256) moments_df_kernel(int64_t nl, int N, const zd* __restrict__ coef,
                                                         void* __restrict__ Y, zd* __restrict__ S) {
    extern __shared__ zdf csf[];  // N x K
    for (int t = threadIdx.x; t < N * K; t += blockDim.x) {
        const zd c = coef[(t / K) + (int64_t)N * (t % K)];
        const float hr = (float)c.re, hi = (float)c.im;
        csf[t] = zdf{hr, hi, (float)(c.re - (double)hr), (float)(c.im - (double)hi)};
    }
    __syncthreads();
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nl) return;
    float rh[K], rl[K], ih[K], il[K];
#pragma unroll
    for (int k = 0; k < K; ++k) rh[k] = rl[k] = ih[k] = il[k] = 0.0f;
    zdf* Yd = reinterpret_cast<zdf*>(Y);
    zd* Yz = reinterpret_cast<zd*>(Y);
    for (int j = 0; j < N; ++j) {
        const zdf y = Yd[(int64_t)j * nl + e];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const zdf c = csf[j * K + k];
            df_fma(rh[k], rl[k], c.hr, c.lr, y.hr, y.lr);    // re += c.re y.re
            df_fms(rh[k], rl[k], c.hi, c.li, y.hi, y.li);    // re -= c.im y.im
            df_fma(ih[k], il[k], c.hr, c.lr, y.hi, y.li);    // im += c.re y.im
            df_fma(ih[k], il[k], c.hi, c.li, y.hr, y.lr);    // im += c.im y.re
        }
        Yz[(int64_t)j * nl + e] = mk((double)y.hr + (double)y.lr, (double)y.hi + (double)y.li);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) S[(int64_t)k * nl + e] = mk((double)rh[k] + (double)rl[k], (double)ih[k] + (double)il[k]);
}

int launch_moments_df(int n, int L, int N, int K, const zd* coef, void* Y, zd* S, cudaStream_t st) {
    const int64_t nl = (int64_t)n * L;
    const int blocks = ceil_div(nl, 256);
    const size_t sm = sizeof(zdf) * (size_t)N * K;
    if (K == 16 && sm <= 96 * 1024) {
        NEP_CUDA(allow_max_dynamic_smem(moments_df_kernel<16>));
        moments_df_kernel<16><<<blocks, 256, sm, st>>>(nl, N, coef, Y, S);
    } else if (K == 8 && sm <= 96 * 1024) {
        NEP_CUDA(allow_max_dynamic_smem(moments_df_kernel<8>));
        moments_df_kernel<8><<<blocks, 256, sm, st>>>(nl, N, coef, Y, S);
    } else {  // other moment counts: Y to FP64, then the FP64 moments
        NEP_TRY(launch_df_to_zd(N, n, L, Y, st));
        return launch_moments(n, L, N, K, coef, reinterpret_cast<const zd*>(Y), S, st);
    }
    NEP_CHECK_LAUNCH();
    return NEP_OK;
}

// mu_k = V^H S_k for all k: one product of V^H (L x n) and the n x (K L) block of the S_k, split over n.
int launch_vh_times(int n, int L, int K, const zd* V, const zd* S, zd* mu, zd* part, size_t part_elems, cudaStream_t st) {
    return zgemm(L, K * L, n, 1, V, n, S, n, mu, L, part, part_elems, st);
}

// H(a*L + i, b*L + c) = mu_{a+b}(i, c), Hs likewise with mu_{a+b+1}; mu_k is L x L column-major.
__global__ void hankel_build_kernel(int L, int M, const zd* __restrict__ mu, zd* __restrict__ H, zd* __restrict__ Hs) {
    const int LM = L * M;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= LM * LM) return;
    const int row = t % LM, colm = t / LM;
    const int a = row / L, i = row % L, b = colm / L, c = colm % L;
    H[t] = mu[(int64_t)(a + b) * L * L + i + (int64_t)L * c];
    Hs[t] = mu[(int64_t)(a + b + 1) * L * L + i + (int64_t)L * c];
}

int launch_hankel_build(int L, int M, const zd* mu, zd* H, zd* Hs, cudaStream_t st) {
    const int LM = L * M;
    hankel_build_kernel<<<ceil_div(LM * LM, 256), 256, 0, st>>>(L, M, mu, H, Hs);
    NEP_CHECK_LAUNCH();
    return NEP_OK;
}


// ------------------------------------------------------------------ conjugate symmetry
// x <- 2 Re x (the sum of a term and its complex conjugate), count entries.
__global__ void double_real_kernel(int64_t count, zd* __restrict__ x) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < count) x[t] = mk(2.0 * x[t].re, 0.0);
}
int launch_double_real(int64_t count, zd* x, cudaStream_t st) {
    if (count <= 0) return NEP_OK;
    double_real_kernel<<<(int)((count + 255) / 256), 256, 0, st>>>(count, x);
    NEP_CHECK_LAUNCH();
    return NEP_OK;
}

// *out = number of entries of x with a nonzero imaginary part.
__global__ void count_imag_kernel(int64_t count, const zd* __restrict__ x, int* __restrict__ out) {
    int c = 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count; t += (int64_t)gridDim.x * blockDim.x)
        c += x[t].im != 0.0;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}
int launch_count_imag(int64_t count, const zd* x, int* out, cudaStream_t st) {
    NEP_CUDA(cudaMemsetAsync(out, 0, sizeof(int), st));
    if (count <= 0) return NEP_OK;
    const int blocks = (int)std::min<int64_t>((count + 255) / 256, 1024);
    count_imag_kernel<<<blocks, 256, 0, st>>>(count, x, out);
    NEP_CHECK_LAUNCH();
    return NEP_OK;
}

}  // namespace nep
