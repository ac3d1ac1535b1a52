// Blocked substitution with complex64 band factors too wide for the register-window sweeps (the
// bandwidth-576 square-root problem): the same forward (row interchanges and unit lower L) and
// backward (upper U, bandwidth kl + ku) sweeps as LAPACK's banded solve, regrouped into blocks of
// NB = 16 steps so that most of the work becomes a small matrix product.
//
// Forward, block of steps c0 .. c0+nb-1, on the window of rows [c0, c0 + nb + kl):
//   * the stored L columns (each taken before the later interchanges of its factorisation) are
//     brought to the block's "panel form": column k takes the interchanges k+1 .. nb-1 of the block
//     (one thread per column). Then M_{nb-1} P_{nb-1} ... M_0 P_0 = M~_{nb-1} ... M~_0 P_{nb-1} ... P_0
//     with M~_k = I - (P_{nb-1} ... P_{k+1} l_k) e_k^T, as no later interchange touches row k;
//   * the block's interchanges are applied to the right-hand sides at once (one thread per column);
//   * the unit lower nb x nb triangle of the panel form gives x (one warp per right-hand side,
//     lane i holding row c0 + i);
//   * the rows below, [c0 + nb, c0 + nb + kl), take w -= L~21 x: a kl x nb by nb x R product, one
//     thread per row with the R right-hand sides in registers.
// Backward, block of rows top .. c1 from the bottom, on the window [top - kl - ku, c1]:
//   * the upper nb x nb triangle gives x (one warp per right-hand side);
//   * the rows above take w -= U(rows, top .. c1) x, U read straight from the band rows; a point without
//     interchanges has ku rows there, not kl + ku.
// The windows are rings of rows in shared memory; rows enter by asynchronous copies into the slots
// the finished block frees, and the next block's L columns and pivots are copied while the current
// block runs. Results equal the sweeps' up to the order of the FP32 roundings.
#include <algorithm>
#include <cstdlib>

#include "band_util.cuh"

namespace nep {

namespace {

constexpr int kBlkNB = 16;     // steps per block
constexpr int kBlkRMax = 16;   // right-hand sides per CTA (register accumulators)
constexpr int kBlkThreads = 512;
constexpr int kBlkChunk = kBlkThreads / 2;  // backward: U rows staged per chunk (two threads a row)
constexpr int kBlkUS = kBlkNB + 1;          // staged U row stride (odd: rows fall on distinct banks)

// RT right-hand-side columns per CTA (a multiple of 4; columns beyond the point's L stay zero).
// Shared memory: X (NB x RT, rows 16-byte aligned for paired loads) first, then the window ring
// (see win), then the forward's two L panels and pivots, or the backward's two U
// triangles and two staged chunks of U rows.
// Element q of window row s: an odd row stride RT + 1, or for RT = 16 rows of 16 rotated by their number, so
// that the lanes of an update (16 rows, both halves) fall in distinct bank pairs either way. Without the
// padding 16 columns fit at bandwidth 576: 64 points x 32 columns are 128 CTAs of 16, one an SM, where 192 of
// 12 ran in two waves (24.8 -> 13.7 ms).
__host__ __device__ constexpr int win_stride(int RT) { return RT == 16 ? 16 : RT + 1; }
template <int RT>
__device__ __forceinline__ int win(int s, int q) {
    return RT == 16 ? s * 16 + ((q + s) & 15) : s * (RT + 1) + q;
}
constexpr size_t kBlkSmemMax = 226 * 1024;
__host__ __device__ inline size_t blk_smem_fwd(int kl, int RT) {
    const size_t PF = kBlkNB + kl;
    return sizeof(zf) * ((size_t)kBlkNB * RT + PF * win_stride(RT) + 2 * (size_t)kBlkNB * PF) + sizeof(int) * 2 * kBlkNB;
}
__host__ __device__ inline size_t blk_smem_bwd(int kv, int RT) {
    const size_t PB = kBlkNB + kv;
    return sizeof(zf) * ((size_t)kBlkNB * RT + PB * win_stride(RT) + 2 * (size_t)kBlkNB * (kBlkNB + 1) +
                         2 * (size_t)kBlkChunk * kBlkUS);
}

// X, the block's solution rows: the columns 2 p and 2 p + 1 of row k as (re, re, im, im)
template <int RT>
__device__ __forceinline__ void x_put(zf* X1, int k, int q, zf v) {
    float* x = reinterpret_cast<float*>(X1 + k * RT + (q & ~1)) + (q & 1);
    x[0] = v.re;
    x[2] = v.im;
}

// Window row s -= sum_k a[k] X[k][..] on one half of the RT columns, two columns per packed multiply-add (the
// operations of fms() in each). Bandwidth 576, 64 points: 16, 24 and 32 columns 10.47, 12.30 and 13.71 -> 10.28,
// 11.95 and 13.28 ms a solve: shared-memory accesses and the copies bound it, not the multiply-adds.
template <int RT>
__device__ __forceinline__ void update_half(zf* W, int s, const zf (&a)[kBlkNB], const zf* X1, int half) {
    constexpr int H = RT / 2, P = H / 2;
    unsigned long long re[P], im[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const zf w0 = W[win<RT>(s, half * H + 2 * p)], w1 = W[win<RT>(s, half * H + 2 * p + 1)];
        re[p] = pack2(w0.re, w1.re);
        im[p] = pack2(w0.im, w1.im);
    }
#pragma unroll
    for (int k = 0; k < kBlkNB; ++k) {
        const ulonglong2* x = reinterpret_cast<const ulonglong2*>(X1 + k * RT + half * H);
        const unsigned long long nr = pack2(-a[k].re, -a[k].re), ai = pack2(a[k].im, a[k].im), ni = pack2(-a[k].im, -a[k].im);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const ulonglong2 v = x[p];
            re[p] = fma2(nr, v.x, re[p]);
            re[p] = fma2(ai, v.y, re[p]);
            im[p] = fma2(nr, v.y, im[p]);
            im[p] = fma2(ni, v.x, im[p]);
        }
    }
#pragma unroll
    for (int p = 0; p < P; ++p) {
        zf w0, w1;
        unpack2(re[p], w0.re, w1.re);
        unpack2(im[p], w0.im, w1.im);
        W[win<RT>(s, half * H + 2 * p)] = w0;
        W[win<RT>(s, half * H + 2 * p + 1)] = w1;
    }
}

template <int RT>
__global__ void __launch_bounds__(kBlkThreads, 1)
    band_solve_blocked_kernel(int n, int kl, int ku, int ldab, const zf* __restrict__ ab_all,
                              const int* __restrict__ ipiv_all, int L, zf* __restrict__ B_all,
                              const int* __restrict__ active) {
    const int j = blockIdx.x;
    if (active && !active[j]) return;
    const int q0 = blockIdx.y * RT;
    const int nr = min(RT, L - q0);
    if (nr <= 0) return;
    constexpr int NB = kBlkNB;
    const int kv = kl + ku;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nthr = blockDim.x, nwarp = nthr >> 5;
    const zf* ab = ab_all + (int64_t)j * n * ldab;
    const int* ipiv = ipiv_all + (int64_t)j * n;
    zf* B = B_all + ((int64_t)j * L + q0) * n;  // right-hand side q at B + q n
    extern __shared__ __align__(16) unsigned char smem_raw[];
    zf* X1 = reinterpret_cast<zf*>(smem_raw);  // NB x RT: the block's solution rows (zero padded)
    zf* sm = X1 + NB * RT;
    const zf zero = mk(0.0f, 0.0f);
    for (int e = tid; e < NB * RT; e += nthr) X1[e] = zero;

    // ===================================================================== forward
    {
        const int PF = NB + kl;
        zf* W = sm;                                 // PF rows: row r at slot r mod PF
        zf* Lp0 = W + (size_t)PF * win_stride(RT);              // 2 x (NB columns of PF local rows)
        int* pv0 = reinterpret_cast<int*>(Lp0 + 2 * (size_t)NB * PF);  // 2 x NB pivots
        auto Lp = [&](int b) { return Lp0 + (size_t)b * NB * PF; };
        for (int e = tid; e < 2 * NB * PF; e += nthr) Lp0[e] = zero;
        for (int q = 0; q < RT; ++q)
            for (int r = tid; r < PF; r += nthr) W[win<RT>(r, q)] = (r < n && q < nr) ? B[(int64_t)q * n + r] : zero;
        __syncthreads();
        // column k of the panel at c0: local rows k+1 .. k+kl from the stored L column c0+k, rows
        // beyond k+kl zero (an earlier block's interchanges may have left values there); rows 0 .. k
        // are never written
        auto issue_panel = [&](int c0, int b) {
            const int nbc = min(NB, n - c0);
            zf* P = Lp(b);
            for (int k = 0; k < nbc; ++k) {
                const zf* src = ab + (int64_t)(c0 + k) * ldab + kv + 1;
                zf* dst = P + (size_t)k * PF + k + 1;
                for (int i = tid; i < kl; i += nthr) cp_async_cx(dst + i, src + i);
            }
            if (tid < NB * NB) {
                const int k = tid / NB, i = tid - k * NB;
                if (i < NB - 1 - k) P[(size_t)k * PF + k + kl + 1 + i] = zero;
            }
            if (tid < nbc) cp_async_i32(&pv0[b * NB + tid], ipiv + c0 + tid);
            cp_async_commit();
        };
        issue_panel(0, 0);
        int sbase = 0;  // slot of row c0
        for (int c0 = 0, blk = 0; c0 < n; c0 += NB, ++blk) {
            const int nbc = min(NB, n - c0);
            const int b = blk & 1;
            cp_async_wait_group<0>();
            __syncthreads();
            if (c0 + NB < n) issue_panel(c0 + NB, b ^ 1);
            zf* P = Lp(b);
            const int* pv = pv0 + b * NB;
            if (tid < nbc) {  // panel form of column k
                zf* col = P + (size_t)tid * PF;
                for (int kp = tid + 1; kp < nbc; ++kp) {
                    const int p = pv[kp] - c0;
                    if (p != kp) {
                        const zf t = col[kp];
                        col[kp] = col[p];
                        col[p] = t;
                    }
                }
            } else if (tid >= 32 && tid < 32 + nr) {  // the block's interchanges, in order
                const int q = tid - 32;
                for (int k = 0; k < nbc; ++k) {
                    const int p = pv[k] - c0;
                    if (p != k) {
                        int s1 = sbase + k, s2 = sbase + p;
                        if (s1 >= PF) s1 -= PF;
                        if (s2 >= PF) s2 -= PF;
                        const zf t = W[win<RT>(s1, q)];
                        W[win<RT>(s1, q)] = W[win<RT>(s2, q)];
                        W[win<RT>(s2, q)] = t;
                    }
                }
            }
            __syncthreads();
            for (int q = warp; q < nr; q += nwarp) {  // unit lower triangle of the panel form
                int s = sbase + lane;
                if (s >= PF) s -= PF;
                zf w = lane < nbc ? W[win<RT>(s, q)] : zero;
                for (int k = 0; k + 1 < nbc; ++k) {
                    const zf xk = shfl_cx(w, k);
                    if (lane > k && lane < nbc) w = fms(w, P[(size_t)k * PF + lane], xk);
                }
                if (lane < NB) x_put<RT>(X1, lane, q, w);  // zero beyond the block's nbc rows
                if (lane < nbc) B[(int64_t)q * n + c0 + lane] = w;
            }
            __syncthreads();
            // rows c0 + PF + i enter the slots of the finished rows c0 + i
            for (int e = tid; e < nbc * nr; e += nthr) {
                const int i = e % nbc, q = e / nbc;
                const int r = c0 + PF + i;
                int s = sbase + i;
                if (s >= PF) s -= PF;
                if (r < n) cp_async_cx(&W[win<RT>(s, q)], B + (int64_t)q * n + r);
                else W[win<RT>(s, q)] = zero;
            }
            cp_async_commit();
            // rows below the block: w -= L~21 x, two threads a row (one half of the columns each);
            // columns of P beyond nbc meet zero rows of X1
            const int rows = min(kl, n - c0 - nbc);
            for (int t = tid; t < 2 * rows; t += nthr) {
                const int lr = nbc + (t >> 1), half = t & 1;
                int s = sbase + lr;
                if (s >= PF) s -= PF;
                zf a[NB];
#pragma unroll
                for (int k = 0; k < NB; ++k) a[k] = P[(size_t)k * PF + lr];
                update_half<RT>(W, s, a, X1, half);
            }
            sbase += nbc;
            if (sbase >= PF) sbase -= PF;
        }
        cp_async_wait_group<0>();
        __syncthreads();
    }

    // ===================================================================== backward
    {
        const int kv = u_reach(n, ku, ipiv);  // this point's U is no wider
        const int PB = NB + kv;
        zf* W = sm;                                  // PB rows: row r at slot r mod PB
        zf* U0 = W + (size_t)PB * win_stride(RT);                // 2 x NB x (NB+1): U(top+i, top+k) at i (NB+1) + k
        zf* S0 = U0 + 2 * (size_t)NB * (NB + 1);     // 2 x kBlkChunk x kBlkUS staged U rows
        auto issue_u11 = [&](int c1, int b) {
            const int top = max(0, c1 - NB + 1), nbc = c1 - top + 1;
            zf* Ub = U0 + (size_t)b * NB * (NB + 1);
            if (tid < NB * NB) {
                const int i = tid / NB, k = tid - i * NB;
                if (i < nbc && k < nbc && k >= i) {
                    if (k - i <= kv) cp_async_cx(&Ub[i * (NB + 1) + k], ab + (int64_t)(top + i) * ldab + (k - i));
                    else Ub[i * (NB + 1) + k] = zero;  // beyond the band (kl + ku < NB - 1)
                }
            }
            cp_async_commit();
        };
        // chunk ch of the block ending at row c1: rows top - kv + ch kBlkChunk + l, their entries
        // U(r, top .. top + NB - 1) (zero beyond the band and beyond the block)
        const int nch = (kv + kBlkChunk - 1) / kBlkChunk;
        auto issue_chunk = [&](int c1, int ch, int b) {
            const int top = max(0, c1 - NB + 1), nbc = c1 - top + 1;
            zf* S = S0 + (size_t)b * kBlkChunk * kBlkUS;
            for (int e = tid; e < kBlkChunk * NB; e += nthr) {
                const int l = e >> 4, k = e & (NB - 1);
                const int t = ch * kBlkChunk + l;
                const int r = top - kv + t;
                const int off = top - r;
                zf* dst = S + l * kBlkUS + k;
                if (t < kv && r >= 0 && k < nbc && off + k <= kv) cp_async_cx(dst, ab + (int64_t)r * ldab + off + k);
                else *dst = zero;
            }
            cp_async_commit();
        };
        for (int q = 0; q < RT; ++q)
            for (int r = max(0, n - PB) + tid; r < n; r += nthr) W[win<RT>(r % PB, q)] = q < nr ? B[(int64_t)q * n + r] : zero;
        for (int e = tid; e < NB * RT; e += nthr) X1[e] = zero;
        issue_u11(n - 1, 0);
        issue_chunk(n - 1, 0, 0);
        int sb = 0;  // staging buffer of the next chunk to compute
        for (int c1 = n - 1, blk = 0; c1 >= 0; c1 -= NB, ++blk) {
            const int top = max(0, c1 - NB + 1), nbc = c1 - top + 1;
            const int b = blk & 1;
            cp_async_wait_group<0>();
            __syncthreads();
            if (top > 0) issue_u11(top - 1, b ^ 1);
            const zf* Ub = U0 + (size_t)b * NB * (NB + 1);
            for (int q = warp; q < nr; q += nwarp) {  // upper triangle, bottom row first
                const zf rd = lane < nbc ? pivot_recip(Ub[lane * (NB + 1) + lane]) : zero;
                zf w = lane < nbc ? W[win<RT>((top + lane) % PB, q)] : zero;
                for (int k = nbc - 1; k >= 0; --k) {
                    const zf xk = shfl_cx(w, k) * shfl_cx(rd, k);
                    if (lane == k) w = xk;
                    else if (lane < k) w = fms(w, Ub[lane * (NB + 1) + k], xk);
                }
                if (lane < NB) x_put<RT>(X1, lane, q, lane < nbc ? w : zero);
                if (lane < nbc) B[(int64_t)q * n + top + lane] = w;
            }
            __syncthreads();
            // rows top - PB + i enter the slots of the finished rows top + i
            for (int e = tid; e < nbc * nr; e += nthr) {
                const int i = e % nbc, q = e / nbc;
                const int r = top - PB + i;
                if (r >= 0) cp_async_cx(&W[win<RT>((top + i) % PB, q)], B + (int64_t)q * n + r);
            }
            cp_async_commit();
            // rows above the block, a chunk of staged U rows at a time: w -= U(r, top .. c1) x
            for (int ch = 0; ch < nch; ++ch) {
                if (ch > 0) {
                    cp_async_wait_group<0>();
                    __syncthreads();
                }
                if (ch + 1 < nch) issue_chunk(c1, ch + 1, sb ^ 1);
                else if (top > 0) issue_chunk(top - 1, 0, sb ^ 1);
                const zf* S = S0 + (size_t)sb * kBlkChunk * kBlkUS;
                const int l = tid >> 1, half = tid & 1;
                const int t = ch * kBlkChunk + l;
                const int r = top - kv + t;
                if (t < kv && r >= 0) {
                    zf a[NB];
#pragma unroll
                    for (int k = 0; k < NB; ++k) a[k] = S[l * kBlkUS + k];
                    update_half<RT>(W, r % PB, a, X1, half);
                }
                sb ^= 1;
            }
        }
        cp_async_wait_group<0>();
    }
}

}  // namespace

// Right-hand sides per CTA (a multiple of 4 up to kBlkRMax whose windows fit in shared memory; 0 if none does):
// the split of a point's columns with the least time, waves of one CTA per SM times 17.5 + columns (bandwidth
// 576, 64 points, ms, before the packed multiply-adds: 16 columns as 2 x 8 10.5, as 16 13.9; 32 as 2 x 16 13.7,
// as 3 x 12 in two waves 24.8).
// The results do not depend on it.
int band_solve_blocked_rhs(int kl, int ku, int npts, int L) {
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 152;
    }();
    int best = 0;
    double least = 0;
    for (int RT = kBlkRMax; RT >= 4; RT -= 4) {
        if (std::max(blk_smem_fwd(kl, RT), blk_smem_bwd(kl + ku, RT)) > kBlkSmemMax) continue;
        const int64_t groups = (L + RT - 1) / RT;
        const double t = (double)(((int64_t)std::max(npts, 1) * groups + sms - 1) / sms) * (17.5 + RT);
        if (best == 0 || t < least) best = RT, least = t;
    }
    return best;
}

template <int RT>
static int launch_blocked(const SplitDev& s, int npts, const zf* ab, const int* ipiv, int L, zf* B, const int* active,
                          cudaStream_t st) {
    const int kv = s.kl + s.ku;
    const size_t smem = std::max(blk_smem_fwd(s.kl, RT), blk_smem_bwd(kv, RT));
    NEP_CUDA(allow_max_dynamic_smem(band_solve_blocked_kernel<RT>));
    dim3 grid(npts, (L + RT - 1) / RT);
    band_solve_blocked_kernel<RT><<<grid, kBlkThreads, smem, st>>>(s.n, s.kl, s.ku, s.ldab, ab, ipiv, L, B, active);
    NEP_CHECK_LAUNCH();
    return NEP_OK;
}

int launch_band_solve_blocked(const SplitDev& s, int npts, const zf* ab, const int* ipiv, int L, zf* B,
                              const int* active, cudaStream_t st) {
    if (npts <= 0 || L <= 0) return NEP_OK;
    switch (band_solve_blocked_rhs(s.kl, s.ku, npts, L)) {
        case 4: return launch_blocked<4>(s, npts, ab, ipiv, L, B, active, st);
        case 8: return launch_blocked<8>(s, npts, ab, ipiv, L, B, active, st);
        case 12: return launch_blocked<12>(s, npts, ab, ipiv, L, B, active, st);
        case 16: return launch_blocked<16>(s, npts, ab, ipiv, L, B, active, st);
        default: return NEP_ERR_UNSUPPORTED;
    }
}

}  // namespace nep
