// The scalar parts of a GMRES cycle, FP64, one warp per Krylov segment (the
// Givens step of a Hessenberg column, the back substitution at its end), and
// the Gram-Schmidt passes of the interface GMRES.
#pragma once

#include "kernels.cuh"

namespace thm {

// Column j of the Hessenberg matrix (h1 + h2 from the two Gram-Schmidt passes,
// ||w|| below the diagonal), previous Givens rotations, a new rotation, the
// updated residual estimate |g_{j+1}| and the per-segment convergence flag.
struct GivensArgs {
    int j, m, ldh;
    const double2* h1;
    const double2* h2;
    double2* Rm;
    double* cs;
    double2* sn;
    double2* gv;
    double2 *pp, *pq, *ip;     // [m+1] p_i, [m] c_i / p_{i+1}, [1] 1 / p_j of the rotations so far (givens_core)
    const double* target;
    int* active;
    int* kused;
    double* beta;
    int* nact;                 // active segments after this step (the first dots pass of the step zeroes it), or null
    int* flag;                 // breakdown (non-finite norm)
    double2* gmon;             // g_{j+1} of segment 0 for the host monitor (single-segment solves), or null
    const int32_t* seg_ch;
    int* cnt;                  // per-segment arrival counters of the last-block reduction
};

__device__ __forceinline__ double2 gv_mul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 gv_fma(double2 a, double2 b, double2 c) {     // a * b + c
    return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}

// One warp.  Applying the previous rotations to the new column is a chain:
// with a_0 = h_0 and, for i < j,
//     r_i     = c_i a_i + s_i h_{i+1}               (entry i of the rotated column)
//     a_{i+1} = A_i a_i + c_i h_{i+1}, A_i = -conj(s_i)  (carried into rotation i + 1).
// With the products p_i = A_0 .. A_{i-1}, which do not depend on the column
// and grow by one factor a step,
//     a_i = p_i (h_0 + sum_{k<i} (c_k / p_{k+1}) h_{k+1}),
// so the chain is a prefix sum over the lanes.  (Every term p_i c_k / p_{k+1}
// is at most 1 in magnitude, so the sum is as stable as the rotations; p_i
// falls like the residual and 1 / p_i is formed beside it, by products.)
// FP64 instructions cost a warp 64 cycles here whatever its active lanes:
// a scan that composes the maps a -> A_i a + B_i took 40 of them where this
// takes 10, and the two square roots run as one on two lanes.  With the scalar
// step's own chain shortened (rsqrt for square root and division, the sums by
// halving, the last step's scalars in shared memory), subdomain solves before
// and after: 2.19 -> 2.07 ms (3^3-cell subdomains), 1.94 -> 1.88 ms (16^2,
// FP64), 4.61 -> 4.53 ms (24^2, order 2).
// Column j of segment s: hin[0..j] (shared memory, unrotated), hn = the
// subdiagonal entry (||w||), ihn = 1 / hn; the rotated column goes to R.
// stop: the segment stops after this column whatever its residual (the last
// column of a cycle).
__device__ bool givens_core(const GivensArgs& ga, int s, int j, const double2* hin, double hn, double ihn, bool stop = false) {
    const int m = ga.m;
    const int lane = threadIdx.x & 31;
    if (!isfinite(hn)) {
        if (lane == 0) {
            atomicExch(ga.flag, 1);
            ga.active[s] = 0;
            ga.beta[s] = 0.0;
        }
        return false;
    }
    const double* cs = ga.cs + (int64_t)s * m;
    const double2* sn = ga.sn + (int64_t)s * m;
    double2* pp = ga.pp + (int64_t)s * (m + 1);
    double2* pq = ga.pq + (int64_t)s * m;
    double2* g = ga.gv + (int64_t)s * (m + 1);
    const double t = ga.target[s];
    const double2 h0 = hin[0], gj = g[j];
    const double2 pj = j > 0 ? pp[j] : make_double2(1, 0), ipj = j > 0 ? ga.ip[s] : make_double2(1, 0);
    const int per = (j + 31) / 32;
    const int b = min(j, lane * per), e = min(j, b + per);
    // the terms of this lane's range, and of the ranges below it
    double2 L = make_double2(0, 0);
    for (int i = b; i < e; ++i) L = gv_fma(pq[i], hin[i + 1], L);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const double2 o = make_double2(__shfl_up_sync(0xffffffffu, L.x, d), __shfl_up_sync(0xffffffffu, L.y, d));
        if (lane >= d) { L.x += o.x; L.y += o.y; }
    }
    double2 S = make_double2(__shfl_up_sync(0xffffffffu, L.x, 1), __shfl_up_sync(0xffffffffu, L.y, 1));
    if (lane == 0) S = make_double2(0, 0);
    S.x += h0.x; S.y += h0.y;                       // a_b / p_b
    double2 a = make_double2(h0.x + __shfl_sync(0xffffffffu, L.x, 31), h0.y + __shfl_sync(0xffffffffu, L.y, 31));
    a = gv_mul(pj, a);                              // a_j
    // the new rotation, from (a_j, ||w||): c = |a| / d, s = (a / |a|) ||w|| / d, d = sqrt(|a|^2 + ||w||^2)
    const double n2a = a.x * a.x + a.y * a.y, d2 = n2a + hn * hn;
    double cj = 1.0;
    double2 sj = make_double2(0, 0);
    const double rs = rsqrt((lane & 1) ? d2 : n2a);
    const double ia = __shfl_sync(0xffffffffu, rs, 0), id = __shfl_sync(0xffffffffu, rs, 1);
    if (n2a == 0.0) {
        if (d2 != 0.0) { cj = 0.0; sj = make_double2(1.0, 0.0); }
    } else {
        const double f = ia * id;
        cj = n2a * f;
        sj = make_double2(a.x * (hn * f), a.y * (hn * f));
    }
    // g_{j+1} = -conj(s) g_j
    const double2 gn = make_double2(-(sj.x * gj.x + sj.y * gj.y), -(sj.x * gj.y - sj.y * gj.x));
    const bool keep = !(stop || gn.x * gn.x + gn.y * gn.y <= t * t || hn == 0.0);
    // the rotated column: rows of this lane's range, and row j
    double2* out = ga.Rm + ((int64_t)s * m + j) * m;
    for (int i = b; i < e; ++i) {
        const double c = cs[i];
        const double2 hi1 = hin[i + 1], p = i > 0 ? pp[i] : make_double2(1, 0), ai = gv_mul(p, S);
        out[i] = gv_fma(sn[i], hi1, make_double2(c * ai.x, c * ai.y));
        if (i + 1 < e) S = gv_fma(pq[i], hi1, S);
    }
    __syncwarp();
    if (lane == 0) {
        out[j] = make_double2(cj * a.x + sj.x * hn, cj * a.y + sj.y * hn);
        ga.cs[(int64_t)s * m + j] = cj;
        ga.sn[(int64_t)s * m + j] = sj;
        g[j + 1] = gn;
        g[j] = make_double2(cj * gj.x, cj * gj.y);
        // p_{j+1} = -conj(s_j) p_j; 1 / conj(s_j) = s_j / |s_j|^2, |s_j| = ||w|| / d
        pp[j + 1] = gv_mul(make_double2(-sj.x, sj.y), pj);
        const double f = n2a == 0.0 ? 1.0 : d2 * ihn * ihn;
        const double2 ip = gv_mul(make_double2(-sj.x * f, -sj.y * f), ipj);
        ga.ip[s] = ip;
        pq[j] = make_double2(cj * ip.x, cj * ip.y);
        if (ga.gmon && s == 0) *ga.gmon = gn;
        ga.kused[s] = j + 1;
        ga.beta[s] = hn;
        if (!keep) ga.active[s] = 0;
        else if (ga.nact) atomicAdd(ga.nact, 1);
    }
    return keep;
}

// Sums NV values per lane over the warp by recursive halving (NV/2 + NV/4 +
// ... + 1 shuffles, then plain ones): lane l ends with the total of value
// l >> (5 - log2 NV).
template <int NV, class R>
__device__ __forceinline__ R warp_sum_many(R (&a)[NV], int lane) {
    int off = 16;
#pragma unroll
    for (int n = NV; n > 1; n >>= 1, off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const R send = up ? a[i] : a[i + n / 2];
            const R keep = up ? a[i + n / 2] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    R v = a[0];
    for (; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// y = R^{-1} g (upper triangular, k columns; R[col * m + row]) by one warp, by
// columns: y_q = g_q / R_qq, then g_i -= R_iq y_q for i < q.  The inverse
// diagonal is formed first and column q - 1 is loaded while column q is used,
// so that no division and no global load is in the chain.  gsh: 2k entries of
// shared memory (the updated g, the inverse diagonal).
__device__ __forceinline__ void backsolve(int m, int k, const double2* R, const double2* gv, double2* gsh, double2* y,
                                          int lane) {
    double2* inv = gsh + k;
    for (int i = lane; i < k; i += 32) {
        gsh[i] = gv[i];
        const double2 d = R[(int64_t)i * m + i];
        const double den = d.x * d.x + d.y * d.y;
        inv[i] = den > 0 ? make_double2(d.x / den, -d.y / den) : make_double2(0, 0);
    }
    constexpr int NP = 4;                      // rows lane, lane + 32, .. of a column in registers
    double2 r[NP];
    auto load = [&](int q) {
#pragma unroll
        for (int p = 0; p < NP; ++p)
            if (lane + 32 * p < q) r[p] = R[(int64_t)q * m + lane + 32 * p];
    };
    load(k - 1);
    __syncwarp();
    for (int q = k - 1; q >= 0; --q) {
        const double2 a = gsh[q], d = inv[q];
        const double2 yq = make_double2(a.x * d.x - a.y * d.y, a.x * d.y + a.y * d.x);
        double2 c[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) c[p] = r[p];
        if (q > 0) load(q - 1);
        if (lane == 0) y[q] = yq;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const int i = lane + 32 * p;
            if (i < q) {
                gsh[i].x = fma(-c[p].x, yq.x, fma(c[p].y, yq.y, gsh[i].x));
                gsh[i].y = fma(-c[p].x, yq.y, fma(-c[p].y, yq.x, gsh[i].y));
            }
        }
        for (int i = lane + 32 * NP; i < q; i += 32) {
            const double2 v = R[(int64_t)q * m + i];
            gsh[i].x = fma(-v.x, yq.x, fma(v.y, yq.y, gsh[i].x));
            gsh[i].y = fma(-v.x, yq.y, fma(-v.y, yq.x, gsh[i].y));
        }
        __syncwarp();
    }
}

constexpr int KW = KT / 32;
constexpr int KSUB = 128;                     // elements that a warp holds, 4 a lane; chunks are multiples of it
constexpr int KEPT = KSUB / 32;

// The last block of a segment to finish (per-segment arrival counter) sums
// the segment's per-chunk partials in chunk order, so the result does not
// depend on which block finishes last, and resets the counter for the next
// launch.  Partials of other blocks are read through L2 (__ldcg).
__device__ __forceinline__ bool last_block_of_segment(int seg, const int32_t* __restrict__ seg_ch, int* cnt) {
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&cnt[seg], 1) == seg_ch[seg + 1] - seg_ch[seg] - 1;
    __syncthreads();
    if (s_last) {
        __threadfence();
        if (threadIdx.x == 0) cnt[seg] = 0;
    }
    return s_last != 0;
}

// Gram-Schmidt passes of the interface GMRES.  A warp works on basis vectors
// of its own (KB at a time, all of a chunk's elements), so a dot product needs
// no sum over the warps, an update one, and a chunk can be as small as 128
// elements: interface systems of a few hundred to ten thousand unknowns spread
// over many SMs.  (Chunks of 1024 elements with the elements shared by the
// warps ran the smaller systems on one SM, whose FP64 units, 2 FMA per clock,
// then worked through zeros, and five rounds of FP64 shuffles a vector; per
// launch, dot products and updates: 256 unknowns 80 -> 16 us and 97 -> 23 us,
// 3-D interfaces of 6^3 cells 124 -> 21 us and 151 -> 29 us.)
constexpr int KB = 4;

// hs[k] += v_k^H w over the elements from e0 on (wr: w of them, by lane), k < nk;
// entry k is one warp's.
__device__ __forceinline__ void sub_chunk_dots(const double2* __restrict__ basis, int64_t ld, int nk, int64_t e0, int64_t end,
                                               const double2 (&wr)[KEPT], double2* hs) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k0 = warp * KB; k0 < nk; k0 += KW * KB) {
        double2 v[KB][KEPT];
#pragma unroll
        for (int b = 0; b < KB; ++b)
#pragma unroll
            for (int q = 0; q < KEPT; ++q) {
                const int64_t e = e0 + lane + 32 * q;
                v[b][q] = k0 + b < nk && e < end ? basis[(int64_t)(k0 + b) * ld + e] : make_double2(0, 0);
            }
        double a[2 * KB];
#pragma unroll
        for (int b = 0; b < 2 * KB; ++b) a[b] = 0;
#pragma unroll
        for (int q = 0; q < KEPT; ++q) {
            if (e0 + 32 * q >= end) break;
#pragma unroll
            for (int b = 0; b < KB; ++b) {
                a[2 * b] = fma(v[b][q].x, wr[q].x, fma(v[b][q].y, wr[q].y, a[2 * b]));         // conj(v) * w
                a[2 * b + 1] = fma(v[b][q].x, wr[q].y, fma(-v[b][q].y, wr[q].x, a[2 * b + 1]));
            }
        }
        const double t = warp_sum_many<2 * KB>(a, lane);     // lane l: value l / 4
        if ((lane & 3) == 0 && k0 + (lane >> 3) < nk) reinterpret_cast<double*>(hs + k0)[lane >> 2] += t;
    }
}

// The segment's h from its chunks' hs (the last block to finish adds them up in chunk order).
__device__ __forceinline__ void chunk_dots_end(const Chunk& c, int nk, const double2* hs, double2* __restrict__ partial, int ldp,
                                               const int32_t* __restrict__ seg_ch, int* __restrict__ cnt,
                                               double2* __restrict__ h, int ldh) {
    __syncthreads();
    for (int kk = threadIdx.x; kk < nk; kk += KT) partial[(int64_t)blockIdx.x * ldp + kk] = hs[kk];
    if (!last_block_of_segment(c.seg, seg_ch, cnt)) return;
    const int c0 = seg_ch[c.seg], c1 = seg_ch[c.seg + 1];
    for (int kk = threadIdx.x; kk < nk; kk += KT) {
        double2 s = make_double2(0, 0);
        constexpr int G = 8;                   // loads in flight
        for (int cc = c0; cc < c1; cc += G) {
            double2 p[G];
#pragma unroll
            for (int g = 0; g < G; ++g) p[g] = cc + g < c1 ? __ldcg(&partial[(int64_t)(cc + g) * ldp + kk]) : make_double2(0, 0);
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (cc + g < c1) s = cadd(s, p[g]);
        }
        h[(int64_t)c.seg * ldh + kk] = s;
    }
}

// w -= sum_k h_k v_k over the KSUB elements from e0 on; the new w of element
// e0 + tid is returned to thread tid < KSUB and kept in sw.  hk: the
// coefficients; sa: [KW][KSUB] sums of the warps.
__device__ __forceinline__ double2 sub_chunk_update(const double2* __restrict__ basis, int64_t ld, int nk, int64_t e0, int64_t end,
                                                    const double2* hk, double2* __restrict__ w, double2* sa, double2* sw) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double2 x[KEPT];
#pragma unroll
    for (int q = 0; q < KEPT; ++q) x[q] = make_double2(0, 0);
    for (int k0 = warp * KB; k0 < nk; k0 += KW * KB) {
        double2 v[KB][KEPT];
#pragma unroll
        for (int b = 0; b < KB; ++b)
#pragma unroll
            for (int q = 0; q < KEPT; ++q) {
                const int64_t e = e0 + lane + 32 * q;
                v[b][q] = k0 + b < nk && e < end ? basis[(int64_t)(k0 + b) * ld + e] : make_double2(0, 0);
            }
#pragma unroll
        for (int q = 0; q < KEPT; ++q) {
            if (e0 + 32 * q >= end) break;
#pragma unroll
            for (int b = 0; b < KB; ++b) {
                const double2 hv = hk[min(k0 + b, nk - 1)];    // beyond nk - 1 the vectors are zeros
                x[q].x = fma(hv.x, v[b][q].x, fma(-hv.y, v[b][q].y, x[q].x));
                x[q].y = fma(hv.x, v[b][q].y, fma(hv.y, v[b][q].x, x[q].y));
            }
        }
    }
#pragma unroll
    for (int q = 0; q < KEPT; ++q) sa[warp * KSUB + lane + 32 * q] = x[q];
    __syncthreads();
    double2 a = make_double2(0, 0);
    if (threadIdx.x < KSUB) {
        const int64_t e = e0 + threadIdx.x;
        if (e < end) {
            const int nw = min(KW, (nk + KB - 1) / KB);        // warps that had vectors
            double2 s = sa[threadIdx.x];
            for (int q = 1; q < nw; ++q) s = cadd(s, sa[q * KSUB + threadIdx.x]);
            a = w[e];
            a = make_double2(a.x - s.x, a.y - s.y);
            w[e] = a;
        }
        sw[threadIdx.x] = a;
    }
    __syncthreads();
    return a;
}

// h[seg][k] = sum over the segment's chunks of v_k^H w, k < nk.
// reset (optional): an int the first block sets to 0 (the active-segment
// count that the Givens step of the same Arnoldi step accumulates).
__global__ void __launch_bounds__(KT) k_chunk_dots(const Chunk* __restrict__ chunks, const double2* __restrict__ basis,
                                                   int64_t ld, int nk, const double2* __restrict__ w,
                                                   double2* __restrict__ partial, int ldp,
                                                   const int* __restrict__ act, const int32_t* __restrict__ seg_ch,
                                                   int* __restrict__ cnt, double2* __restrict__ h, int ldh,
                                                   int* __restrict__ reset, unsigned long long* __restrict__ work) {
    extern __shared__ double2 hs[];            // [nk]
    if (reset && blockIdx.x == 0 && threadIdx.x == 0) *reset = 0;
    const Chunk c = chunks[blockIdx.x];
    if (act && !act[c.seg]) return;            // converged segment: its partials are not read
    if (work && threadIdx.x == 0) atomicAdd(work, (unsigned long long)((nk + 1) * (c.end - c.begin) * sizeof(double2)));
    for (int k = threadIdx.x; k < nk; k += KT) hs[k] = make_double2(0, 0);
    __syncthreads();
    for (int64_t e0 = c.begin; e0 < c.end; e0 += KSUB) {
        double2 wr[KEPT];
#pragma unroll
        for (int q = 0; q < KEPT; ++q) {
            const int64_t e = e0 + (threadIdx.x & 31) + 32 * q;
            wr[q] = e < c.end ? w[e] : make_double2(0, 0);
        }
        sub_chunk_dots(basis, ld, nk, e0, c.end, wr, hs);
    }
    chunk_dots_end(c, nk, hs, partial, ldp, seg_ch, cnt, h, ldh);
}

// First Gram-Schmidt update and second projection in one pass over the
// chunk: w <- w - V h1 (written back), then h2 = V^H w from the updated
// values.  The block rereads its basis slab right after the update, while it
// is in L2, so V is streamed from DRAM once for both.
__global__ void __launch_bounds__(KT) k_update_dots(const Chunk* __restrict__ chunks, const double2* __restrict__ basis,
                                                    int64_t ld, int nk, const double2* __restrict__ h1, int ldh,
                                                    double2* __restrict__ w, double2* __restrict__ partial, int ldp,
                                                    const int* __restrict__ act, const int32_t* __restrict__ seg_ch,
                                                    int* __restrict__ cnt, double2* __restrict__ h2,
                                                    unsigned long long* __restrict__ work) {
    extern __shared__ double2 hk[];            // [nk] coefficients, [nk] dot products
    __shared__ double2 sa[KW * KSUB], sw[KSUB];
    const Chunk c = chunks[blockIdx.x];
    if (act && !act[c.seg]) return;
    // the basis twice, w read and written
    if (work && threadIdx.x == 0) atomicAdd(work, (unsigned long long)((2 * nk + 2) * (c.end - c.begin) * sizeof(double2)));
    double2* hs = hk + nk;
    for (int k = threadIdx.x; k < nk; k += KT) {
        hk[k] = h1[(int64_t)c.seg * ldh + k];
        hs[k] = make_double2(0, 0);
    }
    __syncthreads();
    for (int64_t e0 = c.begin; e0 < c.end; e0 += KSUB) {
        sub_chunk_update(basis, ld, nk, e0, c.end, hk, w, sa, sw);
        double2 wr[KEPT];
#pragma unroll
        for (int q = 0; q < KEPT; ++q) wr[q] = sw[(threadIdx.x & 31) + 32 * q];
        sub_chunk_dots(basis, ld, nk, e0, c.end, wr, hs);
        __syncthreads();                       // sa and sw are written again
    }
    chunk_dots_end(c, nk, hs, partial, ldp, seg_ch, cnt, h2, ldh);
}

}  // namespace thm
