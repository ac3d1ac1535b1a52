// Banded forward/backward substitution (kernel (b), solve part) in blocks of NB = 16 steps.
// Instantiated once per element type (band_subst_f.cu, band_subst_d.cu) so the two compile in
// parallel.
//
// One CTA per (point, RT right-hand sides) runs the forward sweep (row interchanges and unit lower L,
// window of kl rows) and then the backward sweep (U, window of the rows it can reach, ku without
// interchanges and kl + ku at most). Both are written in steps
// s: row s forward, row n-1-s backward; local row i of a block is step s0 + i. A block's coefficients
// form a panel P(i, k), k < 16:
//   forward   P(i, k) = L(c0+i, c0+k), 0 < i - k <= kl, read from ab[(c0+k) ldab + kv + i - k];
//   backward  P(i, k) = U(c1-i, c1-k), 0 <= i - k <= kv, read from ab[(c1-i) ldab + i - k];
// zero outside the band. Rows 0 .. 31 of a panel are its head, the rest its body.
//
// The warps have two roles, joined by one CTA barrier per block:
//   * triangle warps (half a warp per one or two right-hand sides, lane i on row i): in iteration b
//     they take the rows of block b from the window, apply block b-1's solution to them (rows 16 .. 31
//     of head b-1, x by shuffle from the registers that hold it), solve the 16 x 16 triangle (head b;
//     x_k by shuffle, backward times 1/U(c,c)), and publish the solution;
//   * update warps (8): in iteration b they apply block b-1's solution to the window rows beyond
//     block b, w(i) -= sum_k P(i, k) x_k (body b-1): a product of up to kl or kl + ku rows by 16 by RT, each
//     thread keeping TR rows x TQ right-hand sides in registers (TR = 1, 2, 4 by the number of rows). They
//     also stage the panels, the reciprocals of U's diagonal and the rows entering the window.
// So the chain from block to block is one application and one triangle of 16 rows; the long update and
// all loads run beside it. A block with row interchanges takes a slower turn: the stored L columns (each
// taken before the later interchanges of its factorisation) take the block's later interchanges and the
// right-hand sides take all of them (one thread per column). Then
// M_15 P_15 ... M_0 P_0 = M~_15 ... M~_0 P_15 ... P_0, as no later interchange touches row k.
// Every element receives its updates in step order with the operations of the one-step-at-a-time
// sweep, so the results do not depend on RT, TR or the number of stages, bit for bit.
//
// The window is a ring of rows in shared memory. Panel bodies come by cp.async through NS (2 to 4)
// stages, heads four blocks ahead; rows enter the ring NS blocks before their first use. Windows too
// wide for whole backward bodies (kl + ku > 272) stage them in chunks of 256 rows. U is read by rows
// straight from the band: no column copy of U.
//
// What bounds it: the chain from block to block (two barriers' worth of shuffles and 16 dependent
// multiply-adds, 1.8 us a block at bandwidth 64) up to one CTA per SM; beyond that the staging and
// shared-memory instructions of the update, which is why many columns keep the sweeps (band_subst_chosen).
// n = 4096, bandwidth 64, complex64: one right-hand side 0.461 ms (sweeps .661), 64 points x 16 0.612
// (.820); complex128: 9 x 1 3.62 ms (10.6), 64 x 16 6.5 (10.7), bandwidth 40 at 128 x 32 7.5 (11.1);
// bandwidth 200 with interchanges throughout, n = 3000, 16 x 16 9.8 (12.5, one step at a time).
#pragma once
#include <algorithm>
#include <cstdlib>

#include "band_util.cuh"

namespace nep {

namespace subst {
constexpr int NB = 16, UW = 8, NSMAX = 4;
constexpr int HR = 32, HS = 33;   // rows of a head and its stride between columns
constexpr int NHD = 6;            // heads held: blocks b-1 .. b+4
constexpr int RCMAX = 256;        // rows of a staged piece of a backward body

// Right-hand sides per half warp of the triangle warps, and those warps. Complex128: one warp on each of the
// SM's four FP64 units where the registers allow (bandwidth 64, 64 points x 16: 8.47 -> 6.47 ms, 8 right-hand sides
// having kept two units busy and two waiting).
template <typename T>
__host__ __device__ constexpr int tri_rh(int RT) { return RT >= (sizeof(T) == 8 ? 16 : 8) ? 2 : 1; }
template <typename T>
__host__ __device__ constexpr int tri_warps(int RT) { return (RT + 2 * tri_rh<T>(RT) - 1) / (2 * tri_rh<T>(RT)); }
template <typename T>
__host__ __device__ constexpr int threads(int RT) { return 32 * (UW + tri_warps<T>(RT)); }
// Row stride of the window: RT elements, padded to 18 for RT = 16 (two rows x four column groups of 32
// bytes then fall in distinct banks).
__host__ __device__ constexpr int wstride(int RT) { return RT == 16 ? 18 : RT; }
// rows of one staged piece of a body (local rows 32 .. 15 + width); its stride between columns is odd
// (a column's 16 writes spread over the banks)
__host__ __device__ inline int piece_rows(bool bwd, int width) {
    const int body = width > HR - NB ? width - (HR - NB) : 0;
    return bwd && body > RCMAX ? RCMAX : body;
}
__host__ __device__ inline size_t sweep_elems(bool bwd, int width, int RT, int ns) {
    return 2 * (size_t)NB * RT + 2 * NB + (size_t)NHD * NB * HS + (size_t)(width + NB * ns) * wstride(RT) +
           (size_t)ns * NB * (piece_rows(bwd, width) | 1);
}
constexpr size_t PIVBYTES = sizeof(int) * NHD * NB;
// stages that fit in `bytes` of shared memory (0: not even two)
__host__ __device__ inline int stages(bool bwd, int width, int RT, int elem, size_t bytes) {
    for (int ns = NSMAX; ns >= 2; --ns)
        if (elem * sweep_elems(bwd, width, RT, ns) + PIVBYTES <= bytes) return ns;
    return 0;
}
__device__ __forceinline__ void bar_all(int nthreads) { asm volatile("bar.sync 0, %0;" ::"r"(nthreads) : "memory"); }
__device__ __forceinline__ void bar_update() { asm volatile("bar.sync 1, %0;" ::"n"(32 * UW) : "memory"); }
}  // namespace subst

// broadcast of lane k of each half warp
template <typename T>
__device__ __forceinline__ cx<T> shfl16(cx<T> v, int k) {
    cx<T> r;
    r.re = __shfl_sync(0xffffffffu, v.re, k, 16);
    r.im = __shfl_sync(0xffffffffu, v.im, k, 16);
    return r;
}

// w times a reciprocal of U's diagonal. Complex128 with its rounding spelled out: the instances for different
// RT give the same bits.
__device__ __forceinline__ cx<float> mul_diag(cx<float> w, cx<float> rd) { return w * rd; }
__device__ __forceinline__ cx<double> mul_diag(cx<double> w, cx<double> rd) {
    return mk(__fma_rn(w.re, rd.re, -__dmul_rn(w.im, rd.im)), __fma_rn(w.re, rd.im, __dmul_rn(w.im, rd.re)));
}

// TQ consecutive elements from shared memory (pairs of complex64 as one 16-byte load)
template <typename T, int TQ>
__device__ __forceinline__ void ld_row(cx<T> (&v)[TQ], const cx<T>* p) {
    if constexpr (sizeof(T) == 4 && TQ % 2 == 0) {
#pragma unroll
        for (int h = 0; h < TQ / 2; ++h) {
            const float4 f = reinterpret_cast<const float4*>(p)[h];
            v[2 * h] = mk<T>(f.x, f.y);
            v[2 * h + 1] = mk<T>(f.z, f.w);
        }
    } else {
#pragma unroll
        for (int h = 0; h < TQ; ++h) v[h] = p[h];
    }
}
template <typename T, int TQ>
__device__ __forceinline__ void st_row(cx<T>* p, const cx<T> (&v)[TQ]) {
    if constexpr (sizeof(T) == 4 && TQ % 2 == 0) {
#pragma unroll
        for (int h = 0; h < TQ / 2; ++h)
            reinterpret_cast<float4*>(p)[h] = make_float4(v[2 * h].re, v[2 * h].im, v[2 * h + 1].re, v[2 * h + 1].im);
    } else {
#pragma unroll
        for (int h = 0; h < TQ; ++h) p[h] = v[h];
    }
}

// rows [i0, i1) of the window (local indices) -= P X1: warp w takes RGW rows per pass and per t
template <typename T, int RT, int TR>
__device__ __forceinline__ void subst_update(int i0, int i1, int sbase, int PW, cx<T>* W, const cx<T>* P, int SR,
                                             const cx<T>* X1) {
    using namespace subst;
    constexpr int QG = RT >= 4 ? 4 : 1, TQ = RT / QG, RGW = 32 / QG, RTP = wstride(RT);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rl = lane / QG, q0 = (lane % QG) * TQ;
    for (int r0 = i0 + warp * RGW; r0 < i1; r0 += UW * RGW * TR) {
        cx<T> acc[TR][TQ];
        const cx<T>* a[TR];
        cx<T>* w[TR];
        bool ok[TR];
#pragma unroll
        for (int t = 0; t < TR; ++t) {
            int i = r0 + t * UW * RGW + rl;
            ok[t] = i < i1;
            if (!ok[t]) i = i0;
            int s = sbase + i;
            if (s >= PW) s -= PW;
            w[t] = W + s * RTP + q0;
            a[t] = P + i;
            ld_row<T, TQ>(acc[t], w[t]);
        }
#pragma unroll 8
        for (int k = 0; k < NB; ++k) {
            cx<T> x[TQ];
            ld_row<T, TQ>(x, X1 + k * RT + q0);
#pragma unroll
            for (int t = 0; t < TR; ++t) {
                const cx<T> c = a[t][k * SR];
#pragma unroll
                for (int h = 0; h < TQ; ++h) acc[t][h] = fms(acc[t][h], c, x[h]);
            }
        }
#pragma unroll
        for (int t = 0; t < TR; ++t)
            if (ok[t]) st_row<T, TQ>(w[t], acc[t]);
    }
}

template <typename T, int RT, bool BWD>
__device__ __forceinline__ void subst_sweep(int n, int kl, int kv, int ldab, const cx<T>* __restrict__ ab,
                                            const int* __restrict__ ipiv, int nr, cx<T>* B, cx<T>* smem,
                                            size_t smem_bytes) {
    using namespace subst;
    constexpr int RTP = wstride(RT), NT = threads<T>(RT), UT = 32 * UW;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int width = BWD ? kv : kl;
    const int ns = stages(BWD, width, RT, (int)sizeof(cx<T>), smem_bytes);
    const int PW = width + NB * ns;               // ring rows
    const int PR = piece_rows(BWD, width);        // rows per staged piece of a body
    const int SR = PR | 1;
    const int body = max(0, width - (HR - NB));   // rows of a body
    const int nch = PR > 0 ? (body + PR - 1) / PR : 1;  // pieces of a body (1 forward)
    const int nblk = (n + NB - 1) / NB;
    cx<T>* X1 = smem;                             // 2 x NB x RT: the solutions of two blocks
    cx<T>* RD = X1 + 2 * NB * RT;                 // 2 x NB: reciprocals of U's diagonal (backward)
    cx<T>* H0 = RD + 2 * NB;                      // NHD heads of NB x HS
    cx<T>* W = H0 + NHD * NB * HS;                // PW x RTP
    cx<T>* S0 = W + (size_t)PW * RTP;             // ns x NB x SR
    int* piv0 = reinterpret_cast<int*>(S0 + (size_t)ns * NB * SR);  // NHD x NB (forward)
    const cx<T> zero = mk<T>(0, 0);
    auto row_of = [&](int s) { return BWD ? n - 1 - s : s; };

    // Staging (update warps). Every thread's sources move by a fixed distance from block to block, so they
    // are kept as pointers: heads' two entries (hp), the body's first (bp), the entering rows' first (ep).
    const int64_t dblk = BWD ? -(int64_t)NB * ldab : (int64_t)NB * ldab;
    const cx<T>* hp[NB * HR / UT];
    int hdst[NB * HR / UT];  // place in the head, -1: zero there
    int hk[NB * HR / UT], hi[NB * HR / UT];
#pragma unroll
    for (int u = 0; u < NB * HR / UT; ++u) {
        const int e = tid + u * UT;
        hk[u] = BWD ? e & (NB - 1) : (e / HR) & (NB - 1);
        hi[u] = BWD ? (e / NB) & (HR - 1) : e & (HR - 1);
        const int d = hi[u] - hk[u];
        hdst[u] = BWD ? (d >= 0 && d <= kv ? 1 : -1) : (d > 0 && d <= kl ? 1 : -1);
        hp[u] = BWD ? ab + (int64_t)(n - 1 - hi[u]) * ldab + d : ab + (int64_t)hk[u] * ldab + kv + d;
    }
    // head of block b (the next one) into its slot: rows i = 0 .. 31 of the 16 columns
    auto issue_head = [&](int b, int slot) __attribute__((always_inline)) {
        const int left = n - b * NB;  // steps from this block on
        cx<T>* H = H0 + slot * (NB * HS);
#pragma unroll
        for (int u = 0; u < NB * HR / UT; ++u) {
            cx<T>* dst = H + hk[u] * HS + hi[u];
            if (hdst[u] > 0 && hk[u] < left && (!BWD || hi[u] < left)) cp_async_cx(dst, hp[u]);
            else *dst = zero;
            hp[u] += dblk;
        }
        if constexpr (!BWD)
            if (tid < NB && tid < left) cp_async_i32(piv0 + slot * NB + tid, ipiv + b * NB + tid);
    };
    // forward: columns warp and warp + 8, rows 32 + lane on; backward: column tid % 16, rows 32 + tid / 16 on
    const cx<T>* bp = BWD ? ab + (int64_t)(n - 1 - HR - tid / NB) * ldab + (HR + tid / NB) - (tid & (NB - 1))
                          : ab + (int64_t)warp * ldab + kv - warp + HR + lane;
    // piece ch of the body of block b into stage st
    auto issue_body = [&](int b, int ch, int st) __attribute__((always_inline)) {
        const int left = n - b * NB;
        cx<T>* P = S0 + (size_t)st * NB * SR;
        if constexpr (!BWD) {
#pragma unroll
            for (int u = 0; u < NB / UW; ++u) {
                const int k = warp + u * UW;
                const cx<T>* src = bp + (int64_t)u * UW * (ldab - 1);
                cx<T>* dst = P + k * SR + lane;
                const int ie = k < left ? min(body, k + kl + 1 - HR) : 0;  // rows of the body in column k
                for (int i = lane; i < ie; i += 32, src += 32, dst += 32) cp_async_cx(dst, src);
                // zero beyond k + kl (an earlier block's interchanges may have left values there)
                const int z = k + kl + 1 - HR + lane;
                if (lane < NB - 1 - k && z >= 0) P[k * SR + z] = zero;
            }
        } else {
            const int k = tid & (NB - 1), r = tid / NB;
            const int p0 = ch * PR, ie = min(body, p0 + PR);  // rows of the body
            const int last = k < left ? min(ie, min(kv + k + 1 - HR, left - HR)) : 0;
            const cx<T>* src = bp - (int64_t)p0 * (ldab - 1);
            cx<T>* dst = P + k * SR + r;
            for (int i = p0 + r; i < ie; i += UT / NB, src -= (int64_t)(UT / NB) * (ldab - 1), dst += UT / NB) {
                if (i < last) cp_async_cx(dst, src);
                else *dst = zero;
            }
        }
        if (ch == nch - 1) bp += dblk;
    };

    for (int e = tid; e < 2 * NB * RT; e += NT) X1[e] = zero;
    for (int q = 0; q < RT; ++q)
        for (int s = tid; s < PW; s += NT)
            W[s * RTP + q] = (s < n && q < nr) ? B[(int64_t)q * n + row_of(s)] : zero;
    const bool updater = warp < UW;
    if (updater) {
        for (int h = 0; h < NHD - 1; ++h)
            if (h < nblk) issue_head(h, h);
        int b = 0, ch = 0;
        for (int t = 0; t < ns - 1; ++t) {
            if (b < nblk && body > 0) issue_body(b, ch, t);
            cp_async_commit();
            if (++ch == nch) ch = 0, ++b;
        }
        // items (block ib, piece ich) staged next, into stage ist; stage cst is consumed next
        int ib = b, ich = ch, ist = ns - 1, cst = 0;
        int hs = 0;  // head slot of block b
        int sprev = 0;  // ring slot of local row 0 of block b - 1
        const cx<T>* ep = B + (int64_t)(tid / NB) * n + row_of(PW + (tid & (NB - 1)));
        for (b = 0; b < nblk; ++b) {
            auto wait = [&]() {
                if (ns == 2) cp_async_wait_group<0>();
                else if (ns == 3) cp_async_wait_group<1>();
                else cp_async_wait_group<2>();
            };
            wait();
            bar_all(NT);
            bool swaps = false;
            if constexpr (!BWD) {
                const int i = lane & (NB - 1);
                swaps = __any_sync(0xffffffffu, b * NB + i < n && piv0[hs * NB + i] != b * NB + i);
            }
            if (b > 0) {
                const int s0 = (b - 1) * NB;
                const cx<T>* X = X1 + ((b - 1) & 1) * NB * RT;
                const int hn = hs + NHD - 2 >= NHD ? hs - 2 : hs + NHD - 2;  // slot of head b + 4
                for (ch = 0; ch < nch; ++ch) {
                    if (ch > 0) {
                        wait();
                        bar_update();
                    }
                    if (ib < nblk && body > 0) issue_body(ib, ich, ist);
                    if (++ich == nch) ich = 0, ++ib;
                    if (++ist == ns) ist = 0;
                    if (ch == 0) {
                        if (b + NHD - 2 < nblk) issue_head(b + NHD - 2, hn);
                        // steps s0 + PW + i enter the slots of block b - 1 (RT <= 16: one a thread)
                        if (tid < NB * nr) {
                            int s = sprev + (tid & (NB - 1));
                            if (s >= PW) s -= PW;
                            cx<T>* dst = W + s * RTP + tid / NB;
                            if (s0 + PW + (tid & (NB - 1)) < n) cp_async_cx(dst, ep);
                            else *dst = zero;
                        }
                        ep += BWD ? -NB : NB;
                    }
                    cp_async_commit();
                    const int p0 = HR + ch * PR;
                    const int i1 = min(min(NB + width, p0 + PR), n - s0);
                    if (p0 < i1) {
                        constexpr int pass = UW * (RT >= 4 ? 8 : 32);  // rows per pass and TR
                        const cx<T>* P = S0 + (size_t)cst * NB * SR - p0;
                        if (i1 - p0 > 2 * pass) subst_update<T, RT, 4>(p0, i1, sprev, PW, W, P, SR, X);
                        else if (i1 - p0 > pass) subst_update<T, RT, 2>(p0, i1, sprev, PW, W, P, SR, X);
                        else subst_update<T, RT, 1>(p0, i1, sprev, PW, W, P, SR, X);
                    }
                    if (++cst == ns) cst = 0;
                }
                sprev += NB;
                if (sprev >= PW) sprev -= PW;
            }
            const int h1 = hs + 1 == NHD ? 0 : hs + 1;
            if constexpr (BWD) {
                // reciprocals of the next block's diagonal (its head landed one block ahead)
                if (warp == UW - 1 && lane < NB && (b + 1) * NB + lane < n)
                    RD[((b + 1) & 1) * NB + lane] = cdiv(mk<T>(1, 0), H0[h1 * (NB * HS) + lane * HS + lane]);
            } else if (swaps) {
                // the rows of block b are back in the window, its body has landed
                cp_async_wait_group<0>();
                bar_all(NT);
                const int nbc = min(NB, n - b * NB);
                const int* pv = piv0 + hs * NB;
                if (tid < nbc) {
                    cx<T>* H = H0 + hs * (NB * HS) + tid * HS;
                    cx<T>* P = S0 + (size_t)cst * NB * SR + tid * SR - HR;
                    auto at = [&](int i) -> cx<T>& { return i < HR ? H[i] : P[i]; };
                    for (int kp = tid + 1; kp < nbc; ++kp) {
                        const int p = pv[kp] - b * NB;
                        if (p != kp) {
                            const cx<T> v = at(kp);
                            at(kp) = at(p);
                            at(p) = v;
                        }
                    }
                } else if (tid >= 32 && tid < 32 + nr) {
                    const int q = tid - 32;
                    for (int k = 0; k < nbc; ++k) {
                        const int p = pv[k] - b * NB;
                        if (p != k) {
                            int a1 = sprev + k, a2 = sprev + p;
                            if (a1 >= PW) a1 -= PW;
                            if (a2 >= PW) a2 -= PW;
                            const cx<T> v = W[a1 * RTP + q];
                            W[a1 * RTP + q] = W[a2 * RTP + q];
                            W[a2 * RTP + q] = v;
                        }
                    }
                }
                bar_all(NT);
            }
            hs = h1;
        }
    } else {
        constexpr int RH = tri_rh<T>(RT);
        const int i = lane & (NB - 1);
        const int q0 = (2 * (warp - UW) + (lane >> 4)) * RH;  // this half warp's right-hand sides
        const bool live = q0 < RT;
        cx<T>* bo = B + (int64_t)q0 * n + row_of(i);  // this lane's output, block by block
        const int qw = live ? q0 : 0;
        cx<T> x[RH];
#pragma unroll
        for (int h = 0; h < RH; ++h) x[h] = zero;
        int hs = 0, sb = 0;
        // this row's coefficients of block b (triangle) and of block b - 1 on block b (application), read
        // before the barrier that starts iteration b: both heads landed an iteration earlier
        cx<T> pc[NB], pa[NB];
        auto read_triangle = [&](const cx<T>* H) __attribute__((always_inline)) {
#pragma unroll
            for (int k = 0; k < NB; ++k) pc[k] = H[k * HS + i];
        };
#pragma unroll
        for (int k = 0; k < NB; ++k) pa[k] = pc[k] = zero;
        bool first = true;
        for (int b = 0; b < nblk; ++b) {
            const cx<T>* H = H0 + hs * (NB * HS);
            if (!first) read_triangle(H);
            bar_all(NT);
            if (first) read_triangle(H);
            first = false;
            const int nbc = min(NB, n - b * NB);
            bool swaps = false;
            if constexpr (!BWD) swaps = __any_sync(0xffffffffu, i < nbc && piv0[hs * NB + i] != b * NB + i);
            int s = sb + i;
            if (s >= PW) s -= PW;
            cx<T>* wp = W + s * RTP + qw;
            cx<T> w[RH];
            ld_row<T, RH>(w, wp);
            cx<T> rd = zero;
            if constexpr (BWD) {
                if (b > 0) rd = RD[(b & 1) * NB + i];
                else if (i < nbc) rd = cdiv(mk<T>(1, 0), H[i * HS + i]);
            }
            // block b - 1's solution (zero coefficients before the first block)
#pragma unroll
            for (int k = 0; k < NB; ++k)
#pragma unroll
                for (int h = 0; h < RH; ++h) w[h] = fms(w[h], pa[k], shfl16(x[h], k));
            if (!BWD && swaps) {
                if (live) st_row<T, RH>(wp, w);
                bar_all(NT);
                bar_all(NT);
                ld_row<T, RH>(w, wp);
                read_triangle(H);
            }
            // the triangle: lanes below step k keep updating a value that nobody reads
            auto step = [&](int k) __attribute__((always_inline)) {
#pragma unroll
                for (int h = 0; h < RH; ++h) {
                    cx<T> v = w[h];
                    if constexpr (BWD) v = mul_diag(w[h], rd);
                    const cx<T> xk = shfl16(v, k);
                    if (i == k) x[h] = xk;
                    w[h] = fms(w[h], pc[k], xk);
                }
            };
            if (nbc == NB) {
#pragma unroll
                for (int k = 0; k < NB; ++k) step(k);
            } else {
#pragma unroll
                for (int k = 0; k < NB; ++k)
                    if (k < nbc) step(k);
            }
            if (live) {
                cx<T>* X = X1 + (b & 1) * NB * RT + i * RT + q0;
#pragma unroll
                for (int h = 0; h < RH; ++h) {
                    if (i < nbc && q0 + h < nr) {
                        X[h] = x[h];
                        bo[(int64_t)h * n] = x[h];
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < NB; ++k) pa[k] = H[k * HS + NB + i];
            bo += BWD ? -NB : NB;
            hs = hs + 1 == NHD ? 0 : hs + 1;
            sb += NB;
            if (sb >= PW) sb -= PW;
        }
    }
    cp_async_wait_group<0>();
    __syncthreads();
}

template <typename T, int RT>
__global__ void __launch_bounds__(subst::threads<T>(RT), 1)
    band_subst_kernel(int n, int kl, int ku, int ldab, const cx<T>* __restrict__ ab_all,
                      const int* __restrict__ ipiv_all, int L, cx<T>* __restrict__ B_all,
                      const int* __restrict__ active, size_t smem_bytes, const PointDesc* __restrict__ pd) {
    int j = blockIdx.x;
    if (pd) {  // a point of one of several problems sharing the launch (the grid covers the largest L)
        const PointDesc d = pd[blockIdx.x];
        n = d.n, kl = d.kl, ku = d.ku, ldab = d.ldab, L = d.L;
        ab_all = static_cast<const cx<T>*>(d.ab), ipiv_all = d.ipiv;
        B_all = static_cast<cx<T>*>(d.B), active = d.active;
        j = 0;
    }
    if (active && !active[j]) return;
    const int q0 = blockIdx.y * RT;
    const int nr = min(RT, L - q0);
    if (nr <= 0) return;
    const cx<T>* ab = ab_all + (int64_t)j * n * ldab;
    const int* ipiv = ipiv_all + (int64_t)j * n;
    cx<T>* B = B_all + ((int64_t)j * L + q0) * n;  // right-hand side q at B + q n
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T>* smem = reinterpret_cast<cx<T>*>(smem_raw);
    subst_sweep<T, RT, false>(n, kl, kl + ku, ldab, ab, ipiv, nr, B, smem, smem_bytes);
    subst_sweep<T, RT, true>(n, kl, u_reach(n, ku, ipiv), ldab, ab, ipiv, nr, B, smem, smem_bytes);
}

// Shared memory of a launch: what three stages of both sweeps take if two CTAs then share an SM, else
// as many stages as fit one; 0 if the windows do not fit with two stages.
template <typename T>
static size_t subst_smem(int kl, int ku, int RT) {
    const int e = (int)sizeof(cx<T>), kv = kl + ku;
    const size_t half = 113 * 1024, full = 226 * 1024;
    auto need = [&](size_t budget) -> size_t {
        const int nf = subst::stages(false, kl, RT, e, budget), nb = subst::stages(true, kv, RT, e, budget);
        if (!nf || !nb) return 0;
        return e * std::max(subst::sweep_elems(false, kl, RT, nf), subst::sweep_elems(true, kv, RT, nb)) +
               subst::PIVBYTES;
    };
    if (subst::stages(false, kl, RT, e, half) >= 3 && subst::stages(true, kv, RT, e, half) >= 2) return need(half);
    return need(full);
}

// Right-hand sides per CTA (1, 4, 8 or, in FP64, 16; 0: the windows fit with none). solve_rh = 1, 2, 4 (or
// NEP_SOLVE_RH) asks for 4, 8, 16: a launch shape only, the results are identical.
template <typename T>
int band_subst_rt(int kl, int ku, int npts, int L, int rh_force) {
    static const int env = [] {
        const char* e = std::getenv("NEP_SOLVE_RH");
        const int v = e ? std::atoi(e) : 0;
        return (v == 1 || v == 2 || v == 4) ? v : 0;
    }();
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 152;
    }();
    const int rh = rh_force == 1 || rh_force == 2 || rh_force == 4 ? rh_force : env;
    if (L == 1) return subst_smem<T>(kl, ku, 1) ? 1 : 0;
    int want = rh ? 4 * rh : 16;
    if (!rh)
        while (want > 4 && (int64_t)npts * ((L + want - 1) / want) < sms * 3 / 4) want /= 2;
    if (sizeof(T) == 4) want = std::min(want, 8);  // many columns of complex64 take the sweeps
    while (want > 4 && want / 2 >= L) want /= 2;
    for (int rt = want; rt >= 4; rt /= 2)
        if (subst_smem<T>(kl, ku, rt)) return rt;
    return 0;
}

template <typename T, int RT>
static int run_subst(dim3 grid, size_t smem, int n, int kl, int ku, int ldab, const cx<T>* ab, const int* ipiv, int L,
                     cx<T>* B, const int* active, const PointDesc* pd, cudaStream_t st) {
    NEP_CUDA(allow_max_dynamic_smem(band_subst_kernel<T, RT>));
    band_subst_kernel<T, RT><<<grid, subst::threads<T>(RT), smem, st>>>(n, kl, ku, ldab, ab, ipiv, L, B, active, smem, pd);
    NEP_CHECK_LAUNCH();
    return NEP_OK;
}

template <typename T>
static int subst_dispatch(int rt, int npts, int L, size_t smem, int n, int kl, int ku, int ldab, const cx<T>* ab,
                          const int* ipiv, cx<T>* B, const int* active, const PointDesc* pd, cudaStream_t st) {
    const dim3 grid(npts, (L + rt - 1) / rt);
    switch (rt) {
        case 1: return run_subst<T, 1>(grid, smem, n, kl, ku, ldab, ab, ipiv, L, B, active, pd, st);
        case 4: return run_subst<T, 4>(grid, smem, n, kl, ku, ldab, ab, ipiv, L, B, active, pd, st);
        case 8: return run_subst<T, 8>(grid, smem, n, kl, ku, ldab, ab, ipiv, L, B, active, pd, st);
        case 16:
            if constexpr (sizeof(T) == 8) return run_subst<T, 16>(grid, smem, n, kl, ku, ldab, ab, ipiv, L, B, active, pd, st);
    }
    return NEP_ERR_UNSUPPORTED;
}

// T(z_j) X_j = B_j for npts points in place; NEP_ERR_UNSUPPORTED when the windows do not fit.
template <typename T>
int band_subst(const SplitDev& s, int npts, const cx<T>* ab, const int* ipiv, int L, cx<T>* B, const int* active,
               cudaStream_t st, int rh_force) {
    if (npts <= 0 || L <= 0) return NEP_OK;
    const int rt = band_subst_rt<T>(s.kl, s.ku, npts, L, rh_force);
    if (!rt) return NEP_ERR_UNSUPPORTED;
    return subst_dispatch<T>(rt, npts, L, subst_smem<T>(s.kl, s.ku, rt), s.n, s.kl, s.ku, s.ldab, ab, ipiv, B, active,
                             nullptr, st);
}

// The same over points of several problems: rt as band_subst_rt gives it for each of them, smem the
// largest band_subst_smem, pd_dev[count] the descriptors, maxL the most right-hand sides of any.
template <typename T>
size_t band_subst_smem(int kl, int ku, int rt) {
    return subst_smem<T>(kl, ku, rt);
}
template <typename T>
int band_subst_batch(int rt, size_t smem, int count, int maxL, const PointDesc* pd, cudaStream_t st) {
    if (count <= 0 || maxL <= 0) return NEP_OK;
    return subst_dispatch<T>(rt, count, maxL, smem, 0, 0, 0, 0, nullptr, nullptr, nullptr, nullptr, pd, st);
}

#define NEP_INSTANTIATE_SUBST(T)                                                                                      \
    template int band_subst<T>(const SplitDev&, int, const cx<T>*, const int*, int, cx<T>*, const int*, cudaStream_t, \
                               int);                                                                                  \
    template int band_subst_rt<T>(int, int, int, int, int);                                                           \
    template size_t band_subst_smem<T>(int, int, int);                                                                \
    template int band_subst_batch<T>(int, size_t, int, int, const PointDesc*, cudaStream_t);

}  // namespace nep
