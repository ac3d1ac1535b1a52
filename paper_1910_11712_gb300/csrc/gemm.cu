// Dense complex FP64 products C = op(A) B (column-major, op in {A, A^H}) of the extraction: on the tensor core by
// exact 8-bit digit products (oz.cuh), small ones in FP64 FMAs.
//
// Digit products: a CTA of 8 warps computes a 32 x 32 tile, K in blocks of 64: the exponents of the tile's rows and
// columns over the block, then twice 32 terms as digits in the MMA fragments' order in shared memory (A 64 KB, B 32 KB)
// and 36 x 4 MMA steps per warp and 8 x 8 subtile (a warp takes 8 rows by 16 columns); the exact sums of a block
// become FP64 once. Long K splits over CTAs into a workspace reduced in a fixed order, so results never depend
// on scheduling. Blocks with a non-finite entry or an extreme exponent are summed in FP64 FMAs, and so are the
// terms of a block for every result that the guard (oz.cuh) finds too small for the digits.
#include <algorithm>
#include <cmath>

#include "oz.cuh"

namespace nep {

namespace {
constexpr int TB = 32, KH = 32, KCH = KH / 8;  // tile, terms per staged half, MMA steps of a half
constexpr size_t A_WORDS = 4 * KCH * oz::S * 128, B_WORDS = 4 * KCH * oz::S * 64, G_WORDS = 4 * KCH * 64;
}  // namespace

__global__ void __launch_bounds__(256, 2)
    zgemm_oz_kernel(int M, int N, int K, int opA, const zd* __restrict__ A, int lda, const zd* __restrict__ B, int ldb,
                    zd* __restrict__ C, int ldc, int kchunk, int64_t part_stride) {
    using namespace oz;
    extern __shared__ uint4 sm4[];
    unsigned* Af = reinterpret_cast<unsigned*>(sm4);  // [4 row tiles][KCH][S][32 lanes][4]
    unsigned* Bf = Af + A_WORDS;                      // [4 column tiles][KCH][S][32 lanes][2]
    unsigned* Ag = Bf + B_WORDS;                      // [4 row tiles][KCH][32 lanes][2]: the guard's leading bits
    unsigned* Bg = Ag + G_WORDS;                      // [4 column tiles][KCH][32 lanes][2]
    __shared__ int ea[TB], eb[TB], bad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.x * TB, n0 = blockIdx.y * TB;
    const int kb = blockIdx.z * kchunk, ke = min(K, kb + kchunk);
    auto aval = [&](int m, int k) -> zd {
        if (m0 + m >= M || k >= ke) return mk(0.0, 0.0);
        return opA == 0 ? A[m0 + m + (int64_t)lda * k] : conj(A[k + (int64_t)lda * (m0 + m)]);
    };
    auto bval = [&](int c, int k) -> zd { return n0 + c < N && k < ke ? B[k + (int64_t)ldb * (n0 + c)] : mk(0.0, 0.0); };
    const int mt = warp & 3, nt0 = 2 * (warp >> 2);
    // rows and columns of the tile in use, in eights: the rest is neither built nor multiplied
    const int mu = min(TB, (M - m0 + 7) & ~7), nu = min(TB, (N - n0 + 7) & ~7);
    const int g = lane >> 2, tq = lane & 3;
    double out[2][4];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int q = 0; q < 4; ++q) out[u][q] = 0.0;
    for (int k0 = kb; k0 < ke; k0 += CH) {
        const int kn = min(CH, ke - k0);
        __syncthreads();  // the previous block's digits and exponents have been read
        if (tid < TB) ea[tid] = eb[tid] = 0;
        if (tid == 0) bad = 0;
        __syncthreads();
        // lanes along the contiguous index: A by rows (op A) or by k (op A^H), B by k; a warp's 32 entries by k belong
        // to one row or column, and terms beyond the block count as zeros
        for (int e = tid; e < TB * CH; e += 256) {
            const int m = opA == 0 ? e & (TB - 1) : e / CH, k = opA == 0 ? e / TB : e & (CH - 1);
            const int xa = k < kn ? exp_field(aval(m, k0 + k)) : 0;
            if (opA == 0) {
                if (xa) atomicMax(&ea[m], xa);
            } else {
                const int x = __reduce_max_sync(0xffffffffu, xa);
                if (lane == 0 && x) atomicMax(&ea[m], x);
            }
            const int c = e / CH, kk = e & (CH - 1);
            const int xb = __reduce_max_sync(0xffffffffu, kk < kn ? exp_field(bval(c, k0 + kk)) : 0);
            if (lane == 0 && xb) atomicMax(&eb[c], xb);
        }
        __syncthreads();
        if (tid < TB) {
            int x = ea[tid], y = eb[tid];
            if ((x && (x < EXP_LO || x > EXP_HI)) || (y && (y < EXP_LO || y > EXP_HI))) bad = 1;
            if (x == 0) ea[tid] = E_ZERO;
            if (y == 0) eb[tid] = E_ZERO;
        }
        __syncthreads();
        if (bad) {
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int c = 8 * (nt0 + u) + 2 * tq + q;
                    zd acc = mk(out[u][q], out[u][2 + q]);
                    for (int k = 0; k < kn; ++k) acc = fma_(acc, aval(8 * mt + g, k0 + k), bval(c, k0 + k));
                    out[u][q] = acc.re;
                    out[u][2 + q] = acc.im;
                }
            continue;
        }
        float D[2][S][4], G[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int t = 0; t < S; ++t)
#pragma unroll
                for (int q = 0; q < 4; ++q) D[u][t][q] = 0.0f;
        for (int h0 = 0; h0 < kn; h0 += KH) {
            if (h0 > 0) __syncthreads();  // the first half's digits have been read
            for (int e = tid; e < TB * KH; e += 256) {
                const int m = opA == 0 ? e & (TB - 1) : e / KH, k = opA == 0 ? e / TB : e & (KH - 1);
                if (m < mu) {
                    const zd c = aval(m, k0 + h0 + k);
                    const int E = ea[m];
                    const unsigned long long re = fixed62(c.re, E), im = fixed62(c.im, E), ni = fixed62(-c.im, E);
                    unsigned* f = Af + (((m >> 3) * KCH + (k >> 3)) * S) * 128 + ((m & 7) * 4 + (k & 3)) * 4 + ((k & 4) ? 2 : 0);
#pragma unroll
                    for (int t = 0; t < S; ++t)
                        *reinterpret_cast<uint2*>(f + t * 128) =
                            make_uint2(digits2(re, ni, S - 1 - t), digits2(im, re, S - 1 - t));
                    Ag[((m >> 3) * KCH + (k >> 3)) * 64 + ((m & 7) * 4 + (k & 3)) * 2 + ((k & 4) ? 1 : 0)] = lead2(lead(c, E));
                }
                const int c = e / KH;
                if (c < nu) {
                    const int k = e & (KH - 1);
                    const zd y = bval(c, k0 + h0 + k);
                    const int E = eb[c];
                    const unsigned long long re = fixed62(y.re, E), im = fixed62(y.im, E);
                    unsigned* f = Bf + (((c >> 3) * KCH + (k >> 3)) * S) * 64 + ((c & 7) * 4 + (k & 3)) * 2 + ((k & 4) ? 1 : 0);
#pragma unroll
                    for (int t = 0; t < S; ++t) f[t * 64] = digits2(re, im, S - 1 - t);
                    Bg[((c >> 3) * KCH + (k >> 3)) * 64 + ((c & 7) * 4 + (k & 3)) * 2 + ((k & 4) ? 1 : 0)] = lead2(lead(y, E));
                }
            }
            __syncthreads();
            const int kcs = min(KCH, (kn - h0 + 7) / 8);
#pragma unroll 1
            for (int kc = 0; kc < kcs; ++kc) {
                const uint4* a4 = reinterpret_cast<const uint4*>(Af) + (mt * KCH + kc) * S * 32 + lane;
                {  // the guard, columns by rows: one step for the warp's 16 columns
                    const uint2* gb = reinterpret_cast<const uint2*>(Bg) + (nt0 * KCH + kc) * 32 + lane;
                    const uint2 b0 = gb[0], b1 = gb[KCH * 32], a = reinterpret_cast<const uint2*>(Ag)[(mt * KCH + kc) * 32 + lane];
                    mma16816(G, make_uint4(b0.x, b1.x, b0.y, b1.y), a.x, a.y);
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (8 * mt >= mu || 8 * (nt0 + u) >= nu) continue;
                    const uint2* b2 = reinterpret_cast<const uint2*>(Bf) + ((nt0 + u) * KCH + kc) * S * 32 + lane;
                    uint2 b[S];
#pragma unroll
                    for (int t = 0; t < S; ++t) b[t] = b2[t * 32];
#pragma unroll
                    for (int ta = 0; ta < S; ++ta) {
                        const uint4 a = a4[ta * 32];
#pragma unroll
                        for (int tb = 0; ta + tb < S; ++tb) mma16816(D[u][ta + tb], a, b[tb].x, b[tb].y);
                    }
                }
            }
        }
        // columns 2 (lane % 4) + (q & 1); rows lane / 4 (Re for q < 2, else Im)
        const int Ea = ea[8 * mt + g];
        double s[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) s[u][q] = combine(D[u], q, Ea, eb[8 * (nt0 + u) + 2 * tq + (q & 1)]);
#pragma unroll 1
        for (int p = 0; p < 4; ++p) {  // (u, q) = (p / 2, p % 2)
            const int u = p >> 1, q = p & 1, from = 4 * (2 * tq + q) + (g >> 1);  // G's lanes: column lane / 4, rows 2 (lane % 4) + (0, 1)
            const float g0 = __shfl_sync(0xffffffffu, u ? G[2] : G[0], from), g1 = __shfl_sync(0xffffffffu, u ? G[3] : G[1], from);
            const bool weak = ((g & 1) ? g1 : g0) < GUARD && Ea != E_ZERO && eb[8 * (nt0 + u) + 2 * tq + q] != E_ZERO;
            const unsigned todo = __ballot_sync(0xffffffffu, weak);
            if (!todo) continue;
            const zd t = fp64_sums(todo, kn, opA == 0 ? A + m0 + 8 * mt + (int64_t)lda * k0 : A + k0 + (int64_t)lda * (m0 + 8 * mt),
                                   opA == 0 ? 1 : lda, opA == 0 ? lda : 1, opA != 0,
                                   B + k0 + (int64_t)ldb * (n0 + 8 * (nt0 + u) + q), 2 * (int64_t)ldb, 1);
#pragma unroll
            for (int v = 0; v < 4; ++v)
                if (v == p && weak) s[v >> 1][v & 1] = t.re, s[v >> 1][2 + (v & 1)] = t.im;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) out[u][q] += s[u][q];
    }
    zd* Cz = C + (int64_t)blockIdx.z * part_stride;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int gm = m0 + 8 * mt + g, gn = n0 + 8 * (nt0 + u) + 2 * tq + q;
            if (gm < M && gn < N) Cz[gm + (int64_t)ldc * gn] = mk(out[u][q], out[u][2 + q]);
        }
}

// ------------------------------------------------------------------ small products, in FP64 FMAs
// A CTA computes a BM x BN tile with (BM/TM) x (BN/TN) threads of TM x TN outputs, K in steps of GK through shared
// memory; K splits over CTAs into a workspace reduced in a fixed order. The FP64 units bound it (about two FMAs per
// clock per SM), so the launcher picks the tile shape and the split that waste the least of them: padding beyond M
// and N and SMs left idle or doubly loaded.
constexpr int GK = 8;
template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
    zgemm_kernel(int M, int N, int K, int opA, const zd* __restrict__ A, int lda, const zd* __restrict__ B, int ldb,
                 zd* __restrict__ C, int ldc, int kchunk, int64_t part_stride) {
    constexpr int TX = BM / TM, TY = BN / TN, NT = TX * TY;
    __shared__ zd As[GK][BM + 1];
    __shared__ zd Bs[GK][BN + 1];
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    const int kb = blockIdx.z * kchunk, ke = min(K, kb + kchunk);
    zd acc[TM][TN];
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TN; ++b) acc[a][b] = mk(0.0, 0.0);
    for (int k0 = kb; k0 < ke; k0 += GK) {
        // loads run along the contiguous index of each operand
        for (int t = threadIdx.x; t < GK * BM; t += NT) {
            const int kk = opA == 0 ? t / BM : t % GK, mm = opA == 0 ? t % BM : t / GK;
            const int gm = m0 + mm, gk = k0 + kk;
            zd v = mk(0.0, 0.0);
            if (gm < M && gk < ke) v = opA == 0 ? A[gm + (int64_t)lda * gk] : conj(A[gk + (int64_t)lda * gm]);
            As[kk][mm] = v;
        }
        for (int t = threadIdx.x; t < GK * BN; t += NT) {
            const int kk = t % GK, nn = t / GK;
            const int gn = n0 + nn, gk = k0 + kk;
            Bs[kk][nn] = (gn < N && gk < ke) ? B[gk + (int64_t)ldb * gn] : mk(0.0, 0.0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            zd av[TM], bv[TN];
#pragma unroll
            for (int a = 0; a < TM; ++a) av[a] = As[kk][tx + TX * a];
#pragma unroll
            for (int b = 0; b < TN; ++b) bv[b] = Bs[kk][ty + TY * b];
#pragma unroll
            for (int a = 0; a < TM; ++a)
#pragma unroll
                for (int b = 0; b < TN; ++b) acc[a][b] = fma_(acc[a][b], av[a], bv[b]);
        }
        __syncthreads();
    }
    zd* Cz = C + (int64_t)blockIdx.z * part_stride;
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TN; ++b) {
            const int gm = m0 + tx + TX * a, gn = n0 + ty + TY * b;
            if (gm < M && gn < N) Cz[gm + (int64_t)ldc * gn] = acc[a][b];
        }
}

__global__ void zgemm_reduce_kernel(int M, int N, int splits, const zd* __restrict__ part, zd* __restrict__ C, int ldc) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)M * N) return;
    const int m = (int)(t % M), n = (int)(t / M);
    zd acc = mk(0.0, 0.0);
    for (int z = 0; z < splits; ++z) acc = acc + part[(int64_t)z * M * N + t];
    C[m + (int64_t)ldc * n] = acc;
}

namespace {
struct GemmShape {
    int bm, bn;
};
constexpr GemmShape kGemmShapes[] = {{64, 32}, {64, 24}, {32, 32}, {32, 24}, {24, 24}, {32, 16}, {24, 16}};

template <int BM, int BN, int TM, int TN>
void zgemm_launch(dim3 grid, int M, int N, int K, int opA, const zd* A, int lda, const zd* B, int ldb, zd* C, int ldc,
                  int kchunk, int64_t part_stride, cudaStream_t st) {
    zgemm_kernel<BM, BN, TM, TN><<<grid, (BM / TM) * (BN / TN), 0, st>>>(M, N, K, opA, A, lda, B, ldb, C, ldc, kchunk,
                                                                       part_stride);
}
}  // namespace

static int zgemm_fma(int M, int N, int K, int opA, const zd* A, int lda, const zd* B, int ldb, zd* C, int ldc, zd* part,
                     int room, int sms, cudaStream_t st) {
    // score = useful fraction of the padded tiles x SM load balance (mean over max CTAs per SM),
    // a split costing a little for its partial sums and their reduction
    int best = 0, best_splits = 1;
    double best_score = -1.0;
    for (int c = 0; c < (int)(sizeof(kGemmShapes) / sizeof(kGemmShapes[0])); ++c) {
        const int bm = kGemmShapes[c].bm, bn = kGemmShapes[c].bn;
        const int64_t tiles = (int64_t)ceil_div(M, bm) * ceil_div(N, bn);
        const double pad = (double)M * N / ((double)ceil_div(M, bm) * bm * ceil_div(N, bn) * bn);
        const int max_splits = std::max(1, std::min(K / (2 * GK), room));
        for (int sp = 1; sp <= max_splits; ++sp) {
            const double ctas = (double)tiles * sp;
            const double waves = std::ceil(ctas / sms);
            const double score = pad * (ctas / sms) / waves * (sp > 1 ? 0.97 : 1.0);
            if (score > best_score + 1e-9) {
                best_score = score;
                best = c;
                best_splits = sp;
            }
        }
    }
    const int bm = kGemmShapes[best].bm, bn = kGemmShapes[best].bn;
    const int kchunk = ceil_div(ceil_div(K, best_splits), GK) * GK;
    const int splits = std::max(1, ceil_div(K, kchunk));
    dim3 grid(ceil_div(M, bm), ceil_div(N, bn), splits);
    zd* out = splits == 1 ? C : part;
    const int ldo = splits == 1 ? ldc : M;
    const int64_t ps = splits == 1 ? 0 : (int64_t)M * N;
    switch (best) {
        case 0: zgemm_launch<64, 32, 4, 2>(grid, M, N, K, opA, A, lda, B, ldb, out, ldo, kchunk, ps, st); break;
        case 1: zgemm_launch<64, 24, 4, 2>(grid, M, N, K, opA, A, lda, B, ldb, out, ldo, kchunk, ps, st); break;
        case 2: zgemm_launch<32, 32, 2, 2>(grid, M, N, K, opA, A, lda, B, ldb, out, ldo, kchunk, ps, st); break;
        case 3: zgemm_launch<32, 24, 2, 2>(grid, M, N, K, opA, A, lda, B, ldb, out, ldo, kchunk, ps, st); break;
        case 4: zgemm_launch<24, 24, 2, 2>(grid, M, N, K, opA, A, lda, B, ldb, out, ldo, kchunk, ps, st); break;
        case 5: zgemm_launch<32, 16, 2, 1>(grid, M, N, K, opA, A, lda, B, ldb, out, ldo, kchunk, ps, st); break;
        default: zgemm_launch<24, 16, 2, 1>(grid, M, N, K, opA, A, lda, B, ldb, out, ldo, kchunk, ps, st); break;
    }
    NEP_CHECK_LAUNCH();
    if (splits > 1) {
        zgemm_reduce_kernel<<<ceil_div((int64_t)M * N, 256), 256, 0, st>>>(M, N, splits, part, C, ldc);
        NEP_CHECK_LAUNCH();
    }
    return NEP_OK;
}

// FP64 FMAs where the product is small and its K short, or splits to at most 32 terms a CTA: the digits' staging
// and the guard's sums then cost more than they save. us, digits / FMAs, M x N x K: 64 x 21 x 64 28 / 14, 21 x 21 x 21
// (triangular factor: a third of it rejected by the guard) 39 / 14, 9409 x 7 x 7 22 / 11, 66 x 66 x 128 31 / 15, 128 x 66 x 128
// 35 / 22, 96 x 96 x 192 with 192 x 96 x 96 91 / 83; against them 16 x 128 x 64 without room to split 25 / 37,
// 7 x 7 x 9409 48 / 89, 128 x 128 x 128 twice 100 / 103, 4096 x 66 x 66 81 to 91 / 171.
static bool zgemm_small(int M, int N, int K, int max_splits) {
    return K > 0 && (int64_t)M * N * K <= 2000000 && K <= std::min(256, 32 * max_splits);
}

// C = op(A) B. part: workspace of splits*M*N elements when K is long (nullptr => no split).
int zgemm(int M, int N, int K, int opA, const zd* A, int lda, const zd* B, int ldb, zd* C, int ldc, zd* part,
          size_t part_elems, cudaStream_t st) {
    if (M <= 0 || N <= 0) return NEP_OK;
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 152;
    }();
    const int room = part ? std::max(1, (int)std::min<size_t>(64, part_elems / ((size_t)M * N))) : 1;  // splits of K
    if (zgemm_small(M, N, K, room)) return zgemm_fma(M, N, K, opA, A, lda, B, ldb, C, ldc, room > 1 ? part : nullptr, room, sms, st);
    // blocks of 64 terms over as many CTAs as two per SM allow
    const int tiles = ceil_div(M, TB) * ceil_div(N, TB), blocks = std::max(1, ceil_div(K, oz::CH));
    int splits = std::max(1, std::min(std::min(blocks, room), 2 * sms / tiles));
    const int kchunk = ceil_div(blocks, splits) * oz::CH;
    splits = std::max(1, ceil_div(K, kchunk));
    zd* out = splits == 1 ? C : part;
    const int ldo = splits == 1 ? ldc : M;
    const int64_t ps = splits == 1 ? 0 : (int64_t)M * N;
    NEP_CUDA(allow_max_dynamic_smem(zgemm_oz_kernel));
    zgemm_oz_kernel<<<dim3(ceil_div(M, TB), ceil_div(N, TB), splits), 256, sizeof(unsigned) * (A_WORDS + B_WORDS + 2 * G_WORDS), st>>>(
        M, N, K, opA, A, lda, B, ldb, out, ldo, kchunk, ps);
    NEP_CHECK_LAUNCH();
    if (splits > 1) {
        zgemm_reduce_kernel<<<ceil_div((int64_t)M * N, 256), 256, 0, st>>>(M, N, splits, part, C, ldc);
        NEP_CHECK_LAUNCH();
    }
    return NEP_OK;
}

}  // namespace nep
