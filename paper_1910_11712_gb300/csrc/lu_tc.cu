// Kernel (b) for wide bands in complex64: the blocked banded LU of lu_wide.cu with its trailing
// update A22 -= L~21 U12 on the fifth-generation tensor core. One CTA per quadrature point, or a cluster of
// two that share the trailing columns and the operand image.
//
// Elimination, pivot rule and stored factors are those of lu_wide.cu (the unblocked LU's order of
// operations per element); only the trailing product changes arithmetic: it runs as TF32 tensor-
// core products with FP32 accumulation, each FP32 operand split as hi + lo (hi = TF32 rounding,
// lo = TF32 rounding of the rest) and the three products hi*hi + hi*lo + lo*hi summed (~2^-22
// relative error per product, close to FP32; the refinement of the solves removes the rest).
//
// The complex product is one real product (the 4M form): with L~21 = Lr + i Li, U12 = Ur + i Ui,
//   row 2i   of A = [ Lr(i,:)  -Li(i,:) ],  row 2i+1 of A = [ Li(i,:)  Lr(i,:) ],
//   column j of B = [ Ur(:,j) ; Ui(:,j) ],
// so (A B)(2i, j) = Re (L~21 U12)(i, j) and (A B)(2i+1, j) = Im: K = 2 NB = 64, and the real and
// imaginary parts of one complex row sit in adjacent accumulator lanes.
//
// Per panel [p0, p0 + NB):
//   0-1. panel columns to shared memory and factored column by column (as lu_wide.cu);
//   2.   the panel's interchanges on the trailing columns, U12 by forward substitution (a warp per
//        column, lanes over its rows), written back into the window rows p0 .. p0+NB-1 and from
//        there to the output rows;
//   3.   A (from L~21) written to a per-point global operand image in the tensor core's
//        shared-memory layout, 64 complex rows (128 MMA rows) per tile, hi part then lo part;
//   4.   per tile of 128 trailing columns: B (from U12) written to shared memory by the threads;
//        per tile of 64 trailing rows: its A tile staged by a TMA tensor copy (double-buffered),
//        24 MMAs (M = 128, N <= 128, K = 8) into one of two tensor-memory accumulators, and the
//        accumulator drained by all 16 warps (tcgen05.ld), which subtract it from the window.
// The shared memory of steps 0-3 (the panel) and of step 4 (B, two A buffers) is shared.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cooperative_groups.h>
#include <cstdlib>
#include <mutex>
#include <type_traits>

#include "band_util.cuh"
#include "tc_ptx.cuh"

namespace nep {

namespace {
constexpr int NB = 32;                          // panel width: complex columns per panel
constexpr int MT = 64;                          // complex rows per A tile (128 MMA rows)
constexpr int NT = 128;                         // complex columns per B tile (MMA N)
constexpr int KR = 2 * NB;                      // real K of the 4M product
constexpr int PART = 128 * KR;                  // floats in one TF32 part (hi or lo) of a tile
constexpr int TILE_BYTES = 2 * PART * 4;        // hi + lo: 64 KB
constexpr uint32_t LBO = 128 * 16;              // bytes between core matrices adjacent along K
constexpr uint32_t SBO = 128;                   // bytes between 8-row groups
constexpr uint32_t TMEM_COLS = 2 * NT;          // two FP32 accumulators of 128 x 128
constexpr long long WAIT_CYCLES = 4000000000ll; // bounded waits: about two seconds

// (row, k) of a tile -> float offset in one part: core matrices of 8 rows x 4 floats (128 B),
// 16 row groups at SBO, K chunks of 4 at LBO. Inverse: f -> (row, k).
__device__ __forceinline__ void tile_rk(int f, int& r, int& k) {
    const int k4 = f >> 9, rem = f & 511;
    r = (rem >> 5) * 8 + ((rem >> 2) & 7);
    k = k4 * 4 + (rem & 3);
}
}  // namespace

// Scratch beside the panel (step 2): each warp's 8 columns of U12 on their way to the output rows.
namespace {
constexpr int CST = NB + 1, CCOLS = 8;                           // a warp's U12 columns: CCOLS x CST
constexpr size_t STAGE_BYTES = 8 * (size_t)16 * CCOLS * CST;     // 33 KB
// bytes of the region shared by the steps, with the scratch or without
__host__ __device__ inline size_t region_bytes(int kl, bool scratch) {
    const size_t early = 8 * ((size_t)kl + NB) * NB + (scratch ? STAGE_BYTES : 0);
    const size_t late = 3 * (size_t)TILE_BYTES;
    return early > late ? early : late;
}
}  // namespace

static size_t lu_tc_smem_of(int kl, bool scratch) {
    return 1024 + region_bytes(kl, scratch) + sizeof(int) * ((size_t)kl + 2 * NB);
}
// bands whose panel and scratch fit (kl <= 700)
static bool lu_tc_scratch(int kl) { return lu_tc_smem_of(kl, true) <= 224 * 1024; }
size_t lu_tc_smem(int kl) { return lu_tc_smem_of(kl, lu_tc_scratch(kl)); }

// The panel in shared memory with one barrier per column step. Rows stay where they are and carry their
// index as a label: the pivot's label becomes k, row k's label the pivot's. Each warp holds one or two groups
// of 32 rows (all of them for a share of the columns where there are fewer groups than warps); at step k it
// finds the pivot among the groups' candidates, reads the pivot row in place (nobody writes it), and updates
// its rows, column k + 1 first, whose candidates for the next pivot it publishes before the rest. The
// column below the pivot keeps its values, so that every warp can form the multipliers itself; they are
// scaled at the end, when the rows move to their labels' places. The operations per element are those of
// a panel that swaps and scales at every step. At 160 rows the step's chain (pivot search, reciprocal,
// one column) bounds it, not the 31 columns' arithmetic.
constexpr int PW16 = 16;  // warps
// a b, rounded the same wherever it is formed
__device__ __forceinline__ zf mul_cx(zf a, zf b) {
    return mk(__fmaf_rn(a.re, b.re, -__fmul_rn(a.im, b.im)), __fmaf_rn(a.re, b.im, __fmul_rn(a.im, b.re)));
}
template <int NR>  // row groups per warp: 1 (up to 512 rows) or 2
__device__ __forceinline__ void panel_smem(int nbc, int pr, int RW, int kl, int kv, int ldab, int p0, bool writer,
                                           zf* Ps, zf* ab, int* ipiv, int* piv_sh, int* info_s, unsigned (*wkey)[PW16],
                                           int (*wlab)[PW16], int (*wphys)[PW16], int* diag_s, zf* rpv_sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int RG = (RW + 31) / 32;                 // row groups
    const int CG = RG < PW16 ? PW16 / RG : 1;      // shares of the columns
    const int cg = RG < PW16 ? warp / RG : 0;
    const bool on = cg < CG;
    int row[NR], lab[NR];
#pragma unroll
    for (int t = 0; t < NR; ++t) {
        row[t] = t == 0 ? 32 * (RG < PW16 ? warp % RG : warp) + lane : 32 * (warp + PW16) + lane;
        if (!on || row[t] >= RW) row[t] = -1;
        lab[t] = row[t];
    }
    // candidates for pivot k: first row maximising |Re|+|Im| among labels k .. last (no NaN)
    auto publish = [&](int k, const zf (&v)[NR]) __attribute__((always_inline)) {
        const int last = min(k + kl, pr - 1), buf = k & 1;
        unsigned key = 0;
        int cl = 0x7fffffff, ph = 0;
#pragma unroll
        for (int t = 0; t < NR; ++t) {
            if (row[t] < 0 || lab[t] < k || lab[t] > last) continue;
            const float m = abs1(v[t]);
            const unsigned mb = __float_as_uint(m);
            if (m >= 0.0f && (mb > key || (mb == key && lab[t] < cl))) key = mb, cl = lab[t], ph = row[t];
            if (lab[t] == k) diag_s[buf] = row[t];
        }
        const unsigned mx = __reduce_max_sync(0xffffffffu, key);
        const int pl = (int)__reduce_min_sync(0xffffffffu, key == mx ? (unsigned)cl : 0x7fffffffu);
        if (key == mx && cl == pl && pl != 0x7fffffff) wphys[buf][warp] = ph;
        if (lane == 0) wkey[buf][warp] = mx, wlab[buf][warp] = pl;
    };
    if (tid < 2 * PW16) wkey[tid >> 4][tid & 15] = 0, wlab[tid >> 4][tid & 15] = 0x7fffffff;
    __syncthreads();
    if (cg == 0) {
        zf v[NR];
#pragma unroll
        for (int t = 0; t < NR; ++t) v[t] = row[t] >= 0 ? Ps[row[t]] : mk(0.0f, 0.0f);
        publish(0, v);
    }
#pragma unroll 1
    for (int k = 0; k < nbc; ++k) {
        const int last = min(k + kl, pr - 1), buf = k & 1;
        __syncthreads();
        const unsigned key = wkey[buf][lane & 15];
        const int cl = wlab[buf][lane & 15];
        const unsigned mx = __reduce_max_sync(0xffffffffu, key);
        int pl = (int)__reduce_min_sync(0xffffffffu, key == mx ? (unsigned)cl : 0x7fffffffu);
        const unsigned who = __ballot_sync(0xffffffffu, key == mx && cl == pl);
        int ph = wphys[buf][(__ffs(who) - 1) & 15];
        if (pl > last) pl = k, ph = diag_s[buf];  // a column of NaNs: keep the diagonal
        const zf* prow = Ps + ph;
        const zf pv = prow[RW * k];
        const bool zero = pv.re == 0.0f && pv.im == 0.0f;  // then every candidate is zero: pl == k
        const zf rpv = zero ? mk(0.0f, 0.0f) : pivot_recip(pv);
        if (tid == 0) {
            rpv_sh[k] = rpv;
            piv_sh[k] = p0 + pl;
            if (writer) ipiv[p0 + k] = p0 + pl;
            if (zero && *info_s == 0) *info_s = p0 + k + 1;
        }
        zf l[NR];
        bool act[NR];
#pragma unroll
        for (int t = 0; t < NR; ++t) {
            if (row[t] >= 0) lab[t] = lab[t] == pl ? k : lab[t] == k ? pl : lab[t];
            act[t] = row[t] >= 0 && lab[t] > k && lab[t] <= last;
            l[t] = act[t] ? mul_cx(Ps[row[t] + RW * k], rpv) : mk(0.0f, 0.0f);
        }
        if (cg == 0 && k + 1 < nbc) {
            const zf u = prow[RW * (k + 1)];
            zf v[NR];
#pragma unroll
            for (int t = 0; t < NR; ++t) {
                v[t] = mk(0.0f, 0.0f);
                if (row[t] < 0) continue;
                v[t] = Ps[row[t] + RW * (k + 1)];
                if (act[t]) {
                    v[t] = fms(v[t], l[t], u);
                    Ps[row[t] + RW * (k + 1)] = v[t];
                }
            }
            publish(k + 1, v);
        }
        if (on) {
            if (writer && cg == CG - 1) {
                zf* out = ab + (int64_t)(p0 + k) * ldab + kv + 1;
#pragma unroll
                for (int t = 0; t < NR; ++t)
                    if (row[t] >= 0 && lab[t] > k && lab[t] <= k + kl) out[lab[t] - k - 1] = l[t];
            }
#pragma unroll
            for (int t = 0; t < NR; ++t) {
                if (!act[t]) continue;
                const int q0 = k + 1 + (cg == 0 ? CG : cg), st = RW * CG;
                zf* pc = Ps + row[t] + RW * q0;
                const zf* pu = prow + RW * q0;
#pragma unroll 4
                for (int q = q0; q < nbc; q += CG, pc += st, pu += st) *pc = fms(*pc, l[t], *pu);
            }
        }
    }
    __syncthreads();
    // rows to their labels' places, multipliers scaled, half the columns at a time
    int r[NR], d[NR];
#pragma unroll
    for (int t = 0; t < NR; ++t) {
        r[t] = cg == 0 ? row[t] : -1;
        d[t] = lab[t];
    }
#pragma unroll 1
    for (int h = 0; h < NB; h += 8) {
        zf b[NR][8];
#pragma unroll
        for (int t = 0; t < NR; ++t)
            if (r[t] >= 0)
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    b[t][q] = Ps[r[t] + RW * (h + q)];
                    if (h + q < nbc && h + q < d[t]) b[t][q] = mul_cx(b[t][q], rpv_sh[h + q]);
                }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < NR; ++t)
            if (r[t] >= 0)
#pragma unroll
                for (int q = 0; q < 8; ++q) Ps[d[t] + RW * (h + q)] = b[t][q];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(512, 1)
    lu_tc_kernel(int n, int kl, int ku, int ldab, zf* __restrict__ ab_all, int* __restrict__ ipiv_all,
                 int* __restrict__ info_all, const int* __restrict__ active, zf* __restrict__ win_all, int RWp,
                 int CWp, float* __restrict__ aimg_all, int nmt_max, const __grid_constant__ CUtensorMap tmap,
                 int* __restrict__ err, const PointDesc* __restrict__ pd, int passes, int nsplit, int scratch_max_kl) {
    // nsplit CTAs (a cluster) per point: each factors the panel itself and takes its share of the
    // trailing columns; CTA 0 writes the panel's outputs. They build half of the point's operand image each.
    const int j = blockIdx.x / nsplit, part = blockIdx.x - j * nsplit;
    const int img = j;  // operand image and its TMA coordinate
    zf* ab = ab_all + (int64_t)j * n * ldab;
    int* ipiv = ipiv_all + (int64_t)j * n;
    int* info_out = info_all + j;
    zf* W = win_all + (int64_t)j * RWp * CWp;
    if (pd) {  // a point of one of several problems sharing the launch
        const PointDesc d = pd[j];
        n = d.n, kl = d.kl, ku = d.ku, ldab = d.ldab, RWp = d.RWp, CWp = d.CWp;
        ab = static_cast<zf*>(d.ab), ipiv = d.ipiv, info_out = d.info, W = static_cast<zf*>(d.win);
        active = d.active;
        if (active && !active[0]) return;
    } else if (active && !active[j]) {
        return;
    }
    const int kv = kl + ku;
    const int RW = kl + NB;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, nwarp = nthr >> 5;
    float* aimg = aimg_all + (int64_t)img * nmt_max * (TILE_BYTES / 4);
    const bool fast = kl <= scratch_max_kl;  // the scratch fits beside the panel
    // window slots of row p0 + i and column p0 + q of the current panel (rb, cbs: those of p0)
    int rb = 0, cbs = 0;
    auto rs = [&](int i) { return rb + i >= RWp ? rb + i - RWp : rb + i; };
    auto cs_ = [&](int q) { return cbs + q >= CWp ? cbs + q - CWp : cbs + q; };
    auto wi = [&](int i, int q) { return rs(i) + RWp * cs_(q); };

    extern __shared__ unsigned char smem_raw[];
    unsigned char* R = smem_raw + ((1024 - (tc::smem_u32(smem_raw) & 1023)) & 1023);
    zf* Ps = reinterpret_cast<zf*>(R);        // RW x NB panel (steps 0-3)
    float* Bimg = reinterpret_cast<float*>(R);                           // step 4: B (hi, lo)
    float* Abuf0 = reinterpret_cast<float*>(R + TILE_BYTES);             // step 4: A tiles
    float* Abuf1 = reinterpret_cast<float*>(R + 2 * TILE_BYTES);
    zf* scr = Ps + (size_t)RW * NB;           // scratch of steps 1 and 2 (fast)
    int* src = reinterpret_cast<int*>(R + region_bytes(kl, fast));
    int* plist = src + RW;
    __shared__ int piv_sh[NB];
    __shared__ int info_s, npart_s, abort_s, far_s;
    __shared__ zf rpv_sh[NB];
    __shared__ unsigned wkey[2][PW16];
    __shared__ int wlab[2][PW16], wphys[2][PW16], diag_s[2];
    __shared__ uint32_t tmem_s;
    __shared__ __align__(8) uint64_t full_b[2], done_b[2], free_b[2];
    __shared__ int tma_seen[2];

    if (tid == 0) {
        info_s = 0;
        abort_s = 0;
        tma_seen[0] = tma_seen[1] = 0;
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&full_b[b], 1);
            tc::mbar_init(&done_b[b], 1);
            tc::mbar_init(&free_b[b], 16);  // one arrival per warp
        }
        tc::mbar_init_fence();
        tc::tma_prefetch_desc(&tmap);
    }
    if (warp == 0) {
        tc::tmem_alloc(&tmem_s, TMEM_COLS);
        tc::tmem_relinquish();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = tmem_s;
    volatile int* abort_v = &abort_s;
    // bounded wait; a timeout (or an earlier one) sets the error and stops later waits
    auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
        if (*abort_v) return false;
        const long long t0 = clock64();
        while (!tc::mbar_try_wait(bar, parity)) {
            if (*abort_v) return false;
            if (clock64() - t0 > WAIT_CYCLES) {
                *abort_v = 1;
                atomicExch(err, 1);
                return false;
            }
        }
        return true;
    };
    // TMA loads issued into each A buffer (thread 0) and awaited by the MMA issuers
    int tma_issued[2] = {0, 0};
    long long g = 0;  // tiles processed so far: accumulator / A buffer g & 1, phase (g >> 1) & 1

    auto load_rows = [&](int r0, int r1) {
        for (int r = r0 + warp; r < r1; r += nwarp) {
            const zf* srow = ab + (int64_t)r * ldab - (r - kl);  // srow[c] = A(r, c)
            const int clo = max(r - kl, 0), chi = min(r + ku, n - 1);
            for (int c = clo + lane; c <= chi; c += 32) W[wi(r, c)] = srow[c];  // (the first rows: no wrap)
        }
    };
    auto csync = [&]() {  // every CTA of the point: window writes before it are visible after it
        if (nsplit > 1) cooperative_groups::this_cluster().sync();
        else __syncthreads();
    };
    for (int64_t e = tid + (int64_t)part * nthr; e < (int64_t)RWp * CWp; e += (int64_t)nsplit * nthr) W[e] = mk(0.0f, 0.0f);
    csync();
    if (part == 0) load_rows(0, min(RW, n));
    csync();

    int reach = 0;  // last column that a row of U so far can reach: max over the pivots of their row + ku
    for (int p0 = 0; p0 < n; p0 += NB) {
        const int nbc = min(NB, n - p0);
        const int pr = min(RW, n - p0);
        rb = p0 % RWp, cbs = p0 % CWp;

        // ---- 0. panel columns to shared memory (eight independent loads per lane, then the stores)
        for (int q = warp; q < nbc; q += nwarp) {
            const zf* wc = W + RWp * cs_(q);
            for (int i0 = 0; i0 < RW; i0 += 256) {
                zf v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int i = i0 + lane + 32 * u;
                    v[u] = i < pr ? wc[rs(i)] : mk(0.0f, 0.0f);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int i = i0 + lane + 32 * u;
                    if (i < RW) Ps[i + RW * q] = v[u];
                }
            }
        }
        __syncthreads();
        // ---- 1. panel factorisation
        if (RW <= 32 * PW16)
            panel_smem<1>(nbc, pr, RW, kl, kv, ldab, p0, part == 0, Ps, ab, ipiv, piv_sh, &info_s, wkey, wlab, wphys, diag_s, rpv_sh);
        else
            panel_smem<2>(nbc, pr, RW, kl, kv, ldab, p0, part == 0, Ps, ab, ipiv, piv_sh, &info_s, wkey, wlab, wphys, diag_s, rpv_sh);

        // ---- the panel's interchanges as one permutation: local row l receives old row src[l]
        for (int l = tid; l < RW; l += nthr) src[l] = l;
        __syncthreads();
        if (tid == 0) {
            int np = 0, far = 0;
            for (int k = 0; k < nbc; ++k) {
                const int b = piv_sh[k] - p0;
                far = max(far, b);
                if (b != k) {
                    const int t = src[k];
                    src[k] = src[b];
                    src[b] = t;
                    if (b >= nbc) {
                        bool seen = false;
                        for (int q = 0; q < np; ++q) seen |= plist[q] == b;
                        if (!seen) plist[np++] = b;
                    }
                }
            }
            npart_s = np;
            far_s = far;
        }
        __syncthreads();
        const int npart = npart_s;
        // columns beyond the reach are zero in the panel's rows of U, and no row of the panel's interchanges
        // has entries there: the trailing update ends at the reach (kl + ku columns only where rows have
        // traded places; without interchanges bandwidth 128 x 128 points went from 46.6 to 35.6 ms,
        // bandwidth 576 x 64 points from 172 to 121)
        reach = max(reach, p0 + far_s + ku);
        const int cend = min(reach + 1, n), rend = min(p0 + nbc + kl, n);
        const int mr = rend - (p0 + nbc);
        // this CTA's trailing columns [clo, chi)
        const int ctot = cend - (p0 + nbc), cmid = nsplit > 1 ? (ctot / 2 + 15) / 16 * 16 : 0;
        const int clo = p0 + nbc + (part ? min(cmid, ctot) : 0), chi = nsplit > 1 && part == 0 ? p0 + nbc + min(cmid, ctot) : cend;

        // ---- 2. interchanges and U12 = L~11^{-1} A12, one warp per trailing column with lane k on
        // row p0 + k: u_i -= l_ik u_k for k ascending (the substitution's order of operations), the
        // result back into the window rows p0 .. p0+nbc-1 (they retire after this panel)
        // (four columns per warp at a time: four independent substitution chains)
        {
            const int srow = lane < nbc ? src[lane] : 0;
            const int prow = lane < npart ? src[plist[lane]] : 0;
            const int dst = lane < npart ? plist[lane] : 0;
            const zf* lrow = Ps + lane;
            const int wsrc = rs(srow), wprow = rs(prow), wdst = rs(dst), wlane = rs(lane);
            zf* cw = scr + (size_t)warp * CCOLS * CST;
            // eight columns per warp in two groups of four; the next group's loads run ahead
            auto load4 = [&](int q0, zf (&u)[4], zf (&x)[4]) __attribute__((always_inline)) {
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int q = q0 + m;
                    u[m] = q < chi && lane < nbc ? W[wsrc + RWp * cs_(q - p0)] : mk(0.0f, 0.0f);
                    x[m] = q < chi && lane < npart ? W[wprow + RWp * cs_(q - p0)] : mk(0.0f, 0.0f);
                }
            };
            zf u[4], x[4];
            load4(clo + 8 * warp, u, x);
            for (int qb = clo + 8 * warp; qb < chi; qb += 8 * nwarp) {
#pragma unroll
                for (int g4 = 0; g4 < 2; ++g4) {
                    const int q0 = qb + 4 * g4;
                    zf un[4], xn[4];
                    load4(g4 == 0 ? q0 + 4 : qb + 8 * nwarp, un, xn);
                    __syncwarp();  // every lane has read this group's rows
#pragma unroll
                    for (int m = 0; m < 4; ++m)
                        if (q0 + m < chi && lane < npart) W[wdst + RWp * cs_(q0 + m - p0)] = x[m];
                    for (int k = 0; k + 1 < nbc; ++k) {
                        const zf l = lrow[RW * k];
                        const bool act = lane > k && lane < nbc;
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            const zf uk = shfl_cx(u[m], k);
                            if (act) u[m] = fms(u[m], l, uk);
                        }
                    }
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        if (q0 + m < chi && lane < nbc) W[wlane + RWp * cs_(q0 + m - p0)] = u[m];
                        if (fast) cw[(4 * g4 + m) * CST + lane] = u[m];
                    }
#pragma unroll
                    for (int m = 0; m < 4; ++m) u[m] = un[m], x[m] = xn[m];
                }
                if (fast) {  // the eight columns to the output rows: lanes over columns, then rows
                    __syncwarp();
                    const int m = lane & 7, q = qb + m;
#pragma unroll
                    for (int k0 = 0; k0 < NB; k0 += 4) {
                        const int k = k0 + (lane >> 3), r = p0 + k;
                        if (k < nbc && q < chi && q - r <= kv) ab[(int64_t)r * ldab + (q - r)] = cw[m * CST + k];
                    }
                    __syncwarp();
                }
            }
        }
        __syncthreads();
        // U12 rows to the output band (warps over rows, lanes over columns)
        if (!fast)
            for (int k = warp; k < nbc; k += nwarp) {
                const int r = p0 + k;
                for (int q = clo + lane; q < chi; q += 32)
                    if (q - r <= kv) ab[(int64_t)r * ldab + (q - r)] = W[wi(k, q - p0)];
            }

        // ---- the panel part of the finished rows: U(r, r .. p0+nbc-1), zeros beyond the band
        for (int k = part == 0 ? warp : nbc; k < nbc; k += nwarp) {
            const int r = p0 + k;
            zf* out = ab + (int64_t)r * ldab;
            for (int q = k + lane; q < nbc; q += 32) out[q - k] = Ps[k + (int64_t)RW * q];
            for (int t = (cend - r) + lane; t <= kv; t += 32)
                if (t >= 0) out[t] = mk(0.0f, 0.0f);
        }

        // ---- 3. A operand image of L~21 (global, the tensor core's layout), tiles of 64 rows
        const int nmt = mr > 0 ? (mr + MT - 1) / MT : 0;
        const int ntn = (chi > clo && mr > 0) ? (chi - clo + NT - 1) / NT : 0;
        if (ctot > 0 && nmt > 0) {
            const int mine = (nmt - part + nsplit - 1) / nsplit;  // tiles part, part + nsplit, ...
            for (int e = tid; e < mine * PART; e += nthr) {
                const int mt = e / PART * nsplit + part, f = e % PART;
                int r, k;
                tile_rk(f, r, k);
                const int i = mt * MT + (r >> 1), cc = k & (NB - 1);
                float v = 0.0f;
                if (i < mr && cc < nbc) {
                    const zf l = Ps[nbc + i + (int64_t)RW * cc];
                    const bool imrow = (r & 1) != 0, second = k >= NB;
                    v = imrow ? (second ? l.re : l.im) : (second ? -l.im : l.re);
                }
                float hi, lo;
                tc::split_tf32(v, hi, lo);
                float* t = aimg + (int64_t)mt * 2 * PART;
                t[f] = hi;
                t[PART + f] = lo;
            }
            tc::fence_async_global();
        }
        csync();
        if (nsplit > 1) tc::fence_async_global();  // the other CTA's half, before this one's copies read it

        // ---- 4. A22 -= L~21 U12 on the tensor core
        for (int nt = 0; nt < ntn; ++nt) {
            const int c0 = clo + nt * NT;
            const int ncol = min(NT, chi - c0), ncol16 = (ncol + 15) & ~15;  // the product's N
            const uint32_t idesc = tc::idesc_tf32(128, ncol16);
            if (tid == 0 && !*abort_v)
                for (int q = 0; q < min(2, nmt); ++q) {
                    const int b = (int)((g + q) & 1);
                    float* dst = b ? Abuf1 : Abuf0;
                    tc::mbar_arrive_expect_tx(&full_b[b], TILE_BYTES);
                    tc::tma_load_3d(dst, &tmap, &full_b[b], 0, q * 256, img);
                    ++tma_issued[b];
                }
            // the C rows of the first A tile towards L2 while B is built (lane q: column q of its group)
            if ((warp >> 2) * 32 + lane < ncol && 16 * (warp & 3) < mr)
                tc::prefetch_l2(W + wi(nbc + 16 * (warp & 3), c0 - p0 + (warp >> 2) * 32 + lane));
            // B: row rn of the operand = complex column c0 + rn of U12, K = [Ur ; Ui]; lanes over the
            // 32 rows of U12 (contiguous in the window), eight independent loads, then the stores
            for (int e0 = 0; e0 < NB * NT; e0 += 8 * nthr) {
                zf u[8];
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    const int e = e0 + tid + s * nthr, kk = e & (NB - 1), rn = e >> 5;
                    u[s] = rn < ncol && kk < nbc ? W[wi(kk, c0 - p0 + rn)] : mk(0.0f, 0.0f);
                }
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    const int e = e0 + tid + s * nthr, kk = e & (NB - 1), rn = e >> 5;
                    if (rn >= ncol16) break;  // a whole warp's
                    const int fr = (kk >> 2) * 512 + (rn >> 3) * 32 + (rn & 7) * 4 + (kk & 3);  // k = kk
                    const int fi = fr + (NB >> 2) * 512;                                        // k = kk + NB
                    float hi, lo;
                    tc::split_tf32(u[s].re, hi, lo);
                    Bimg[fr] = hi;
                    Bimg[PART + fr] = lo;
                    tc::split_tf32(u[s].im, hi, lo);
                    Bimg[fi] = hi;
                    Bimg[PART + fi] = lo;
                }
            }
            tc::fence_async_shared();
            __syncthreads();

            // MMA issue for tile t of this column tile: one lane, of another warp for every tile, since it
            // comes to its part of the window about 1.5 us later than the rest (bandwidth 576, 64 points: the
            // update 126 -> 86 us a panel, the factorisation 117 -> 97 ms; with thread 0 issuing every
            // product, each tile waited for its warp)
            auto issue = [&](int t) {
                const long long gt = g + t;
                const int b = (int)(gt & 1);
                if (!wait(&full_b[b], (uint32_t)((gt >> 1) & 1))) return;
                atomicAdd(&tma_seen[b], 1);
                if (gt >= 2 && !wait(&free_b[b], (uint32_t)(((gt >> 1) - 1) & 1))) return;
                tc::tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(b * NT);
                const uint32_t abase = tc::smem_u32(b ? Abuf1 : Abuf0), bbase = tc::smem_u32(Bimg);
                // passes = 3: hi*hi + hi*lo + lo*hi (~FP32); passes = 1: hi*hi alone (TF32 operands).
                // (the start address is the descriptor's low field, in 16 bytes: steps add to it)
                const uint64_t ad = tc::smem_desc(abase, LBO, SBO), bd = tc::smem_desc(bbase, LBO, SBO);
                constexpr uint64_t step = 2 * LBO / 16, lo = PART * 4 / 16;
#pragma unroll
                for (int s = 0; s < KR / 8; ++s) tc::mma_tf32(d, ad + s * step, bd + s * step, idesc, s != 0);
                if (passes == 3) {
#pragma unroll
                    for (int s = 0; s < KR / 8; ++s) tc::mma_tf32(d, ad + s * step, bd + lo + s * step, idesc, 1);
#pragma unroll
                    for (int s = 0; s < KR / 8; ++s) tc::mma_tf32(d, ad + lo + s * step, bd + s * step, idesc, 1);
                }
                tc::mma_commit(&done_b[b]);
            };
            for (int t = 0; t < nmt; ++t) {
                const long long gt = g + t;
                const int b = (int)(gt & 1);
                const uint32_t ph = (uint32_t)((gt >> 1) & 1);
                const int cb = (warp >> 2) * 32;  // this warp's 32 columns of the tile
                // the C rows of tile t + 1 towards L2: lane q takes column cb + q, one line (16 rows)
                if (t + 1 < nmt && cb + lane < ncol) {
                    const int i = (t + 1) * MT + 16 * (warp & 3);
                    if (i < mr)
                        tc::prefetch_l2(W + wi(nbc + i, c0 - p0 + cb + lane));
                }
                if (tid == 0 && t == 0) issue(0);
                if (lane == 0 && t + 1 < nmt && warp == (int)((gt + 1) & 15)) issue(t + 1);
                __syncwarp();
                const bool ok = __all_sync(0xffffffffu, wait(&done_b[b], ph));
                // MMA t is done: its A buffer takes tile t + 2 (the copy runs during this epilogue)
                if (tid == 0 && ok && t + 2 < nmt) {
                    float* dst = b ? Abuf1 : Abuf0;
                    tc::mbar_arrive_expect_tx(&full_b[b], TILE_BYTES);
                    tc::tma_load_3d(dst, &tmap, &full_b[b], 0, (t + 2) * 256, img);
                    ++tma_issued[b];
                }
                __syncwarp();
                if (ok && cb >= ncol) {
                    if (lane == 0) tc::mbar_arrive(&free_b[b]);
                } else if (ok) {
                    tc::tc_fence_after();
                    float v[32];
                    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b * NT + cb);
                    tc::tmem_ld_32x32b_x32(taddr, v);
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&free_b[b]);
                    // lanes 2m and 2m+1 hold the real and imaginary rows of complex row m: they trade
                    // halves, the even lane then updating columns 0..15 and the odd one 16..31 as
                    // complex (8-byte) read-modify-writes
                    const bool odd = (lane & 1) != 0;
                    float re[16], im[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const float send = odd ? v[q] : v[16 + q];
                        const float recv = __shfl_xor_sync(0xffffffffu, send, 1);
                        re[q] = odd ? recv : v[q];
                        im[q] = odd ? v[16 + q] : recv;
                    }
                    const int rr = (warp & 3) * 32 + lane;
                    const int i = t * MT + (rr >> 1);
                    if (i < mr) {
                        zf* wrow = W + rs(nbc + i);
                        const int h = odd ? 16 : 0;
                        const int cs = cs_(c0 - p0 + cb + h);
                        zf cur[16];
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            const int sl = cs + q < CWp ? cs + q : cs + q - CWp;
                            cur[q] = cb + h + q < ncol ? wrow[(int64_t)RWp * sl] : mk(0.0f, 0.0f);
                        }
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            const int sl = cs + q < CWp ? cs + q : cs + q - CWp;
                            if (cb + h + q < ncol) wrow[(int64_t)RWp * sl] = mk(cur[q].re - re[q], cur[q].im - im[q]);
                        }
                    }
                }
            }
            g += nmt;
            __syncthreads();
        }
        if (*abort_v) break;

        // ---- 5. next window: rows [p0+RW, p0+RW+NB) and columns [p0+RW.., ) enter
        if (nsplit > 1) csync();  // the other CTA is done with the rows and columns that leave
        if (p0 + NB < n) {
            const int CW = kv + NB;
            const int rn0 = p0 + RW;
            const int nws = nwarp * nsplit, wid = part * nwarp + warp;  // warps of all CTAs
            for (int jc = wid; jc < NB; jc += nws) {
                zf* wc = W + RWp * ((p0 + CW + jc) % CWp);
                for (int i = lane; i < RWp; i += 32) wc[i] = mk(0.0f, 0.0f);
            }
            csync();
            // column slot s holds the column c in [p0 + NB, p0 + NB + CWp) with c = s (mod CWp)
            const int r = rn0 + lane, rslot = r % RWp;
            const int per = (CWp + nws - 1) / nws;
            const int cbase = p0 + NB, cb0 = cbase % CWp, send = min(CWp, (wid + 1) * per);
            for (int s0 = wid * per; s0 < send; s0 += 8) {
                zf v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int s = s0 + u;
                    const int c = cbase + (s < cb0 ? s - cb0 + CWp : s - cb0);
                    v[u] = (s < send && lane < NB && r < n && c >= r - kl && c <= r + ku && c < n)
                               ? ab[(int64_t)r * ldab + (c - r + kl)]
                               : mk(0.0f, 0.0f);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int s = s0 + u;
                    if (s < send) W[rslot + RWp * s] = v[u];
                }
            }
        }
        csync();
    }
    // wind down: copies and products in flight finish (bounded) before the memory is released
    if (tid == 0) {
        for (int b = 0; b < 2; ++b)
            for (int u = tma_seen[b]; u < tma_issued[b]; ++u) {
                const long long t0 = clock64();
                while (!tc::mbar_try_wait(&full_b[b], (uint32_t)(u & 1)) && clock64() - t0 < WAIT_CYCLES) {
                }
            }
        if (g > 0) {
            const long long last = g - 1;
            const long long t0 = clock64();
            while (!tc::mbar_try_wait(&done_b[last & 1], (uint32_t)((last >> 1) & 1)) && clock64() - t0 < WAIT_CYCLES) {
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, TMEM_COLS);
    }
    if (tid == 0 && part == 0) *info_out = *abort_v ? n + 1 : info_s;
}

// ------------------------------------------------------------------ host side
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

bool lu_tc_enabled() {
    static const bool on = [] {
        const char* e = getenv("NEP_LU_TC");
        return !(e && e[0] == '0');
    }();
    return on;
}

// CTAs per point: two where the device then still holds every CTA at once. Both factor the whole panel: latency
// bought with work. A pass alone takes 41.1 ms with two and 42.8 with one at bandwidth 97, 155 and 204 at 576 (64 points
// each); with other passes on the device one CTA gives the higher throughput: bandwidth 97, 8 pipelines, 29.7 and 23.6 ms
// a pass, though at 576 with 2 pipelines two still lead, 132 and 150.
static int lu_tc_split(int npts) {
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 152;
    }();
    return 2 * npts <= sms ? 2 : 1;
}
// the largest kl with the scratch
static int lu_tc_scratch_max_kl() {
    static const int v = [] {
        int kl = 0;
        while (lu_tc_scratch(kl + 1)) ++kl;
        return kl;
    }();
    return v;
}
template <typename... Args>
static cudaError_t lu_tc_start(int npts, int nsplit, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(npts * nsplit);
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = nsplit;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, lu_tc_kernel, args...);
}

// The panel of kl rows fits the shared memory that a launch may ask for: what a CTA can have less the kernel's
// static part (kl <= 854; wider bands take lu_wide.cu)
bool band_lu_tc_can(int kl) {
    static const size_t room = [] {
        cudaFuncAttributes a{};
        const cudaError_t e = cudaFuncGetAttributes(&a, lu_tc_kernel);
        if (e != cudaSuccess) cudaGetLastError();  // no device: nothing is launched
        return (size_t)smem_optin_bytes() - (e == cudaSuccess ? a.sharedSizeBytes : 1024);
    }();
    return kl >= NB && lu_tc_smem(kl) <= room;
}

bool band_lu_tc_fits(int kl) { return kl > 64 && band_lu_tc_can(kl); }

int launch_band_lu_tc(const SplitDev& s, int npts, zf* ab, int* ipiv, int* info, const int* active, cudaStream_t st,
                      int passes) {
    if (npts <= 0) return NEP_OK;
    if (!band_lu_tc_can(s.kl)) return NEP_ERR_UNSUPPORTED;
    auto encode = encode_fn();
    if (!encode) {
        set_error("cuTensorMapEncodeTiled is not available from the driver");
        return NEP_ERR_CUDA;
    }
    const int kv = s.kl + s.ku;
    const int rwp = (s.kl + NB + NB - 1) / NB * NB, cwp = (kv + NB + NB - 1) / NB * NB;
    const size_t smem = lu_tc_smem(s.kl);
    const int nmt_max = (s.kl + MT - 1) / MT, nsplit = lu_tc_split(npts);
    zf* win = nullptr;
    float* aimg = nullptr;
    int* err = nullptr;
    NEP_CUDA(cudaMallocAsync((void**)&win, sizeof(zf) * (size_t)rwp * cwp * npts, st));
    cudaError_t e = cudaMallocAsync((void**)&aimg, (size_t)TILE_BYTES * nmt_max * npts, st);
    if (e == cudaSuccess) e = cudaMallocAsync((void**)&err, sizeof(int), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), st);
    CUtensorMap tmap;
    if (e == cudaSuccess) {
        // the operand images as a 3-D array of floats: 64 per image row (256 B), 256 image rows per
        // tile, nmt_max tiles per point, npts points; one box = one tile (64 KB)
        const cuuint64_t dims[3] = {64, (cuuint64_t)nmt_max * 256, (cuuint64_t)npts};
        const cuuint64_t strides[2] = {256, (cuuint64_t)nmt_max * TILE_BYTES};
        const cuuint32_t box[3] = {64, 256, 1};
        const cuuint32_t estr[3] = {1, 1, 1};
        const CUresult r = encode(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, aimg, dims, strides, box, estr,
                                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            cudaFreeAsync(win, st);
            cudaFreeAsync(aimg, st);
            cudaFreeAsync(err, st);
            set_error("cuTensorMapEncodeTiled failed (%d)", (int)r);
            return NEP_ERR_CUDA;
        }
    }
    if (e == cudaSuccess) e = allow_max_dynamic_smem(lu_tc_kernel);
    if (e == cudaSuccess) {
        e = lu_tc_start(npts, nsplit, smem, st, s.n, s.kl, s.ku, s.ldab, ab, ipiv, info, active, win, rwp, cwp, aimg,
                        nmt_max, tmap, err, (const PointDesc*)nullptr, passes, nsplit, lu_tc_scratch_max_kl());
        count_launch();
    }
    int herr = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (win) cudaFreeAsync(win, st);
    if (aimg) cudaFreeAsync(aimg, st);
    if (err) cudaFreeAsync(err, st);
    if (e != cudaSuccess) return cuda_fail(e, "lu_tc_kernel", __FILE__, __LINE__);
    if (herr) {
        set_error("lu_tc_kernel: a bounded wait on the tensor-core pipeline expired");
        return NEP_ERR_INTERNAL;
    }
    return NEP_OK;
}

// The tensor-core LU over points of several complex64 problems (each with kl > 64 and within the
// shared-memory budget): windows per point, one operand-image array and tensor map for the batch.
int launch_band_lu_tc_batch(const std::vector<PointDesc>& items_in, cudaStream_t st, int passes) {
    const int count = (int)items_in.size();
    if (count <= 0) return NEP_OK;
    auto encode = encode_fn();
    if (!encode) {
        set_error("cuTensorMapEncodeTiled is not available from the driver");
        return NEP_ERR_CUDA;
    }
    std::vector<PointDesc> items(items_in);
    size_t smem = 0, win_elems = 0;
    int nmt_max = 1;
    const int nsplit = lu_tc_split(count);
    for (auto& d : items) {
        if (!band_lu_tc_can(d.kl)) return NEP_ERR_UNSUPPORTED;
        const int kv = d.kl + d.ku;
        d.RWp = (d.kl + NB + NB - 1) / NB * NB;
        d.CWp = (kv + NB + NB - 1) / NB * NB;
        win_elems += (size_t)d.RWp * d.CWp;
        smem = std::max(smem, lu_tc_smem(d.kl));
        nmt_max = std::max(nmt_max, (d.kl + MT - 1) / MT);
    }
    zf* win = nullptr;
    float* aimg = nullptr;
    int* err = nullptr;
    PointDesc* pd = nullptr;
    NEP_CUDA(cudaMallocAsync((void**)&win, sizeof(zf) * win_elems, st));
    cudaError_t e = cudaMallocAsync((void**)&aimg, (size_t)TILE_BYTES * nmt_max * count, st);
    if (e == cudaSuccess) e = cudaMallocAsync((void**)&err, sizeof(int), st);
    if (e == cudaSuccess) e = cudaMallocAsync((void**)&pd, sizeof(PointDesc) * count, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), st);
    size_t off = 0;
    for (auto& d : items) {
        d.win = win + off;
        off += (size_t)d.RWp * d.CWp;
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(pd, items.data(), sizeof(PointDesc) * count, cudaMemcpyHostToDevice, st);
    CUtensorMap tmap;
    if (e == cudaSuccess) {
        const cuuint64_t dims[3] = {64, (cuuint64_t)nmt_max * 256, (cuuint64_t)count};
        const cuuint64_t strides[2] = {256, (cuuint64_t)nmt_max * TILE_BYTES};
        const cuuint32_t box[3] = {64, 256, 1};
        const cuuint32_t estr[3] = {1, 1, 1};
        if (encode(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, aimg, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            e = cudaErrorInvalidValue;
    }
    if (e == cudaSuccess) e = allow_max_dynamic_smem(lu_tc_kernel);
    if (e == cudaSuccess) {
        e = lu_tc_start(count, nsplit, smem, st, 0, 0, 0, 0, (zf*)nullptr, (int*)nullptr, (int*)nullptr, (const int*)nullptr,
                        (zf*)nullptr, 0, 0, aimg, nmt_max, tmap, err, (const PointDesc*)pd, passes, nsplit,
                        lu_tc_scratch_max_kl());
        count_launch();
    }
    int herr = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (win) cudaFreeAsync(win, st);
    if (aimg) cudaFreeAsync(aimg, st);
    if (err) cudaFreeAsync(err, st);
    if (pd) cudaFreeAsync(pd, st);
    if (e != cudaSuccess) return cuda_fail(e, "lu_tc_kernel (batch)", __FILE__, __LINE__);
    if (herr) {
        set_error("lu_tc_kernel: a bounded wait on the tensor-core pipeline expired");
        return NEP_ERR_INTERNAL;
    }
    return NEP_OK;
}

}  // namespace nep
