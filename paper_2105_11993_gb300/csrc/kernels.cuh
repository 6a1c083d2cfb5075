// Device kernels of the solve phase (templated on vector/value precision).
#pragma once

#include "common.cuh"

namespace thm {

template <class V> struct VT;
template <> struct VT<double2> { using R = double; };
template <> struct VT<float2> { using R = float; };

template <class V>
__device__ __forceinline__ V mk(typename VT<V>::R a, typename VT<V>::R b);
template <> __device__ __forceinline__ double2 mk<double2>(double a, double b) { return make_double2(a, b); }
template <> __device__ __forceinline__ float2 mk<float2>(float a, float b) { return make_float2(a, b); }

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// ---------------------------------------------------------------------------
// y = T_i x  (op 0: P + i(B_Gamma + B_Sigma))  or  K_i^loc x (op 2: P + i B_Gamma)
// SELL-32: one thread per row, slots column-major inside a slice (coalesced).
// ---------------------------------------------------------------------------
// 3-D: the face terms are not diagonal; their values (times kappa*omega) ride
// on the same SELL pattern (bvg: Gamma^inf, bvs: Sigma), non-null only then.
// Column indices: int32 local indices, or (CI = uint16_t) indices relative
// to the row's subdomain (origin: its first local row), half the bytes of the
// index stream.  xs: x at the column origin.
// The matrix arrays of one precision.
template <class F>
struct SpmvMat {
    const F *val, *bg, *bs;
    const F *bvg, *bvs;       // 3-D only
};
// Row r times x: slots in groups of 8, so that the 8 index and value loads,
// then the 8 gathers of x, are in flight together.
template <class V, class F, class CI>
__device__ __forceinline__ V spmv_row(int64_t r, const int64_t* __restrict__ slice_ptr, const CI* __restrict__ col,
                                      const SpmvMat<F>& A, int use_bs, const V* xs, int64_t origin) {
    using R = typename VT<V>::R;
    const int64_t base = __ldg(slice_ptr + (r >> 5));
    const int w = (int)((__ldg(slice_ptr + (r >> 5) + 1) - base) >> 5);
    const int64_t at = base + (r & 31);
    const CI* cp = col + at;
    const F* vp = A.val + at;
    R ar = 0, ai = 0;
    if (A.bvg) {
        const F* gp = A.bvg + at;
        const F* sp = A.bvs + at;
        for (int t = 0; t < w; ++t) {
            const int32_t c = (int32_t)__ldg(cp + (t << 5));
            const R v = (R)__ldg(vp + (t << 5));
            R b = (R)__ldg(gp + (t << 5));
            if (use_bs) b += (R)__ldg(sp + (t << 5));
            const V xv = xs[c];
            ar += v * xv.x - b * xv.y;
            ai += v * xv.y + b * xv.x;
        }
    } else {
        for (int t0 = 0; t0 < w; t0 += 8) {
            int32_t c[8];
            R v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                c[u] = (int32_t)(r - origin);      // own row (its x is read below anyway)
                v[u] = 0;
                if (t0 + u < w) {
                    c[u] = (int32_t)__ldg(cp + ((t0 + u) << 5));
                    v[u] = (R)__ldg(vp + ((t0 + u) << 5));
                }
            }
            V xv[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) xv[u] = xs[c[u]];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                ar += v[u] * xv[u].x;
                ai += v[u] * xv[u].y;
            }
        }
    }
    R b = (R)__ldg(A.bg + r);
    if (use_bs) b += (R)__ldg(A.bs + r);
    const V xr = xs[r - origin];
    return mk<V>(ar - b * xr.y, ai + b * xr.x);
}

template <class V, class F, class CI = int32_t>
__global__ void __launch_bounds__(256) k_spmv(int64_t n, const int64_t* __restrict__ slice_ptr,
                                              const CI* __restrict__ col, const Sub* __restrict__ subs,
                                              SpmvMat<F> A, int use_bs, const V* __restrict__ x,
                                              V* __restrict__ y, const int32_t* __restrict__ row_seg,
                                              unsigned long long* __restrict__ work) {
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (work) {                                // rows processed (uniform branch: every thread reaches the count)
        const int cnt = __syncthreads_count(r < n);
        if (threadIdx.x == 0 && cnt) atomicAdd(work, (unsigned long long)cnt);
    }
    if (r >= n) return;
    int64_t origin = 0;
    if constexpr (sizeof(CI) == 2) origin = subs[row_seg[r]].off;
    y[r] = spmv_row<V, F, CI>(r, slice_ptr, col, A, use_bs, x + origin, origin);
}

// ---- TMA 1-D bulk copies completing on an mbarrier (sm_90+ PTX) ----------
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// bytes must be a multiple of 16, both addresses 16-byte aligned
__device__ __forceinline__ void tma_load_1d(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// Segmented passes over vectors.  A chunk lies inside one segment (a problem
// of a batch); per-chunk partials are summed per segment in a
// fixed order, so every dot product is deterministic.
// ---------------------------------------------------------------------------
constexpr int KT = 256;                       // threads per chunk block

template <class V>
__global__ void __launch_bounds__(KT) k_chunk_norm2(const Chunk* __restrict__ chunks, const V* __restrict__ x,
                                                    double* __restrict__ nrm_part) {
    using R = typename VT<V>::R;
    __shared__ double sw[KT / 32];
    const Chunk c = chunks[blockIdx.x];
    R nr = 0;
    for (int64_t e = c.begin + threadIdx.x; e < c.end; e += KT) {
        V v = x[e];
        nr += v.x * v.x + v.y * v.y;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nr += __shfl_down_sync(0xffffffffu, nr, o);
    if (lane == 0) sw[warp] = (double)nr;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int q = 0; q < KT / 32; ++q) s += sw[q];
        nrm_part[blockIdx.x] = s;
    }
}

__global__ void k_seg_reduce_real(int nseg, const int32_t* __restrict__ seg_ch, const double* __restrict__ part,
                                  double* __restrict__ out);

// scale: x[e] = (beta[seg] > 0) ? r[e] / beta[seg] : 0, and 0 in segments that are not active (act, or null)
template <class V>
__global__ void k_chunk_scale(const Chunk* __restrict__ chunks, const V* __restrict__ r,
                              const double* __restrict__ beta, V* __restrict__ x, const int* __restrict__ act) {
    using R = typename VT<V>::R;
    __shared__ R s_inv;
    const Chunk c = chunks[blockIdx.x];
    if (act && !act[c.seg]) {                  // the operator runs over all segments
        for (int64_t e = c.begin + threadIdx.x; e < c.end; e += blockDim.x) x[e] = mk<V>(0, 0);
        return;
    }
    if (threadIdx.x == 0) {                    // one FP64 division per block, not per thread
        const double b = beta[c.seg];
        s_inv = b > 0 ? (R)(1.0 / b) : (R)0;
    }
    __syncthreads();
    const R inv = s_inv;
    for (int64_t e = c.begin + threadIdx.x; e < c.end; e += blockDim.x) {
        V v = r[e];
        x[e] = mk<V>(v.x * inv, v.y * inv);
    }
}

// t[e] = sum_{k < kused[seg]} y[seg][k] basis_k[e]
template <class V>
__global__ void __launch_bounds__(KT) k_chunk_combine(const Chunk* __restrict__ chunks, const V* __restrict__ basis,
                                                      int64_t ld, const int* __restrict__ kused,
                                                      const double2* __restrict__ y, int ldy, V* __restrict__ t) {
    using R = typename VT<V>::R;
    extern __shared__ double2 ys_raw[];        // [ldy] y of this segment in the vector precision
    V* ys = reinterpret_cast<V*>(ys_raw);
    const Chunk c = chunks[blockIdx.x];
    const int nk = kused[c.seg];
    const double2* yy = y + (int64_t)c.seg * ldy;
    for (int k = threadIdx.x; k < nk; k += KT) ys[k] = mk<V>((R)yy[k].x, (R)yy[k].y);
    __syncthreads();
    for (int64_t e = c.begin + threadIdx.x; e < c.end; e += KT) {
        R xr = 0, xi = 0;
        for (int k = 0; k < nk; ++k) {
            const V v = basis[(int64_t)k * ld + e], a = ys[k];
            xr += a.x * v.x - a.y * v.y;
            xi += a.x * v.y + a.y * v.x;
        }
        t[e] = mk<V>(xr, xi);
    }
}

template <class V>
__global__ void k_axpy(int64_t n, const V* __restrict__ a, V* __restrict__ x) {  // x += a
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) {
        V u = x[i], v = a[i];
        x[i] = mk<V>(u.x + v.x, u.y + v.y);
    }
}

template <class V>
__global__ void k_sub(int64_t n, const V* __restrict__ a, const V* __restrict__ b, V* __restrict__ out) {  // a - b
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) {
        V u = a[i], v = b[i];
        out[i] = mk<V>(u.x - v.x, u.y - v.y);
    }
}

}  // namespace thm
