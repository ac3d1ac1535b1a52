// Kernel (a): split-form assembly of the shifted matrices T(z_j) = sum_i f_i(z_j) A_i
// (Sec. 2 Eq. (split); Sec. 3.2.2 builds T(lambda) from the f_i values and l-1 sparse
// axpys) for every quadrature point at once, written straight into the row-oriented band
// storage that the banded LU consumes.
//
// One warp per point and kAsmRows rows: it zero-fills the rows' slots with 16-byte stores, then its lanes
// run over the rows' union-pattern entries, consecutive in the pattern, and write
// sum_i F[i,j] a_i(r,k) (FP64 sum, one rounding to the storage type) to slot k - r + kl. The FP64 row sums of
// |t_rk| give ||T(z_j)||_inf for the refinement's backward error; the FP64 values of T(z_j) on the
// union pattern (tval) feed the residual of the refinement.
// Bound: HBM writes (n*ldab elements per point), or the FP64 units when there is no band to write: an FP64
// instruction costs the same for one lane as for 32, and a warp per row left 27 of 32 idle with five-point
// patterns. n = 16384, five-point,
// bandwidth 128, 128 points: 4.31 -> 1.24 ms with the band (6.5 GB written).
#include "nep_common.cuh"

namespace nep {

__device__ __forceinline__ void atomic_max_nonneg(double* addr, double v) {
    // non-negative doubles order like their bit patterns
    atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}

constexpr int kAsmRows = 16;

// count elements of zero from p on, by one warp
template <typename T>
__device__ __forceinline__ void warp_zero(cx<T>* p, int64_t count, int lane) {
    if constexpr (sizeof(T) == 4) {
        if (reinterpret_cast<uintptr_t>(p) & 15) {
            if (lane == 0 && count > 0) p[0] = mk<T>(0, 0);
            ++p, --count;
        }
        float4* q = reinterpret_cast<float4*>(p);
        for (int64_t t = lane; t < count / 2; t += 32) q[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lane == 0 && (count & 1) && count > 0) p[count - 1] = mk<T>(0, 0);
    } else {
        for (int64_t t = lane; t < count; t += 32) p[t] = mk<T>(0, 0);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) assemble_band_kernel(SplitDev s, int npts, const zd* __restrict__ F,
                                                            cx<T>* __restrict__ ab, double* __restrict__ tnorm,
                                                            zd* __restrict__ tval) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int groups = (s.n + kAsmRows - 1) / kAsmRows;
    if (gw >= (int64_t)npts * groups) return;
    const int j = (int)(gw / groups);
    const int r0 = (int)(gw - (int64_t)j * groups) * kAsmRows, nrows = min(kAsmRows, s.n - r0);
    cx<T>* band = ab ? ab + ((int64_t)j * s.n + r0) * s.ldab : nullptr;
    if (band) warp_zero(band, (int64_t)nrows * s.ldab, lane);
    __syncwarp();
    // lane q holds the first entry of row r0 + q (of the row past the group from nrows on)
    const int64_t first = s.rowptr[r0 + min(lane, nrows)], last = __shfl_sync(0xffffffffu, first, nrows);
    const int64_t next = __shfl_down_sync(0xffffffffu, first, 1);
    double rowsum = 0.0;  // of row r0 + lane
    for (int64_t e0 = __shfl_sync(0xffffffffu, first, 0); e0 < last; e0 += 32) {
        const int64_t e = e0 + lane;
        int q = -1;  // the entry's row
        for (int t = 0; t < nrows; ++t) q += e >= __shfl_sync(0xffffffffu, first, t);
        double mod = 0.0;
        if (e < last) {
            zd v = mk(0.0, 0.0);
            for (int i = 0; i < s.nterms; ++i) {
                zd f = F[i + (int64_t)s.nterms * j];
                zd a = mk(s.val[(int64_t)i * s.nnz + e], s.val_im ? s.val_im[(int64_t)i * s.nnz + e] : 0.0);
                v = fma_(v, f, a);
            }
            if (band) band[(int64_t)q * s.ldab + (s.col[e] - (r0 + q) + s.kl)] = cvt<T>(v);
            if (tval) tval[(int64_t)j * s.nnz + e] = v;
            if (tnorm) mod = hypot(v.re, v.im);
        }
        if (tnorm) {  // each row's lane adds the row's entries in their order
            const int64_t lo = lane < nrows ? max(first, e0) : 0, hi = lane < nrows ? min(next, e0 + 32) : 0;
            const int most = __reduce_max_sync(0xffffffffu, (int)max(hi - lo, (int64_t)0));
            for (int t = 0; t < most; ++t) {
                const double m = __shfl_sync(0xffffffffu, mod, (int)(lo + t - e0) & 31);
                if (lo + t < hi) rowsum += m;
            }
        }
    }
    if (tnorm) {
        long long top = __double_as_longlong(rowsum);  // sums order like their bits, a NaN above all
        for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        if (lane == 0) atomic_max_nonneg(tnorm + j, __longlong_as_double(top));
    }
}

template <typename T>
int launch_assemble(const SplitDev& s, int npts, const zd* F, cx<T>* ab, double* tnorm, zd* tval, cudaStream_t st) {
    if (npts <= 0) return NEP_OK;
    if (tnorm) NEP_CUDA(cudaMemsetAsync(tnorm, 0, sizeof(double) * npts, st));
    const int64_t warps = (int64_t)npts * ((s.n + kAsmRows - 1) / kAsmRows);
    const int blocks = ceil_div(warps * 32, 256);
    assemble_band_kernel<T><<<blocks, 256, 0, st>>>(s, npts, F, ab, tnorm, tval);
    NEP_CHECK_LAUNCH();
    return NEP_OK;
}

template int launch_assemble<float>(const SplitDev&, int, const zd*, cx<float>*, double*, zd*, cudaStream_t);
template int launch_assemble<double>(const SplitDev&, int, const zd*, cx<double>*, double*, zd*, cudaStream_t);

}  // namespace nep
