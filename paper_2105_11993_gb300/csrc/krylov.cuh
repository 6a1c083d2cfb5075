// The scalar parts of a GMRES cycle, FP64, one warp per Krylov segment: the
// Givens step of a Hessenberg column and the back substitution at its end.
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
//     a_{i+1} = -conj(s_i) a_i + c_i h_{i+1}         (carried into rotation i + 1)
// the carry follows the affine maps a -> A_i a + B_i (A_i = -conj(s_i),
// B_i = c_i h_{i+1}), which compose associatively.  Each lane composes the
// maps of its range of i, a shuffle scan gives every lane the composition of
// the ranges below it (so its incoming carry), and the lanes then walk their
// ranges in parallel.  FP64 instructions cost a full warp slot on this part
// whatever the active lanes, so the serial chain of about 12 of them per
// rotation on one lane becomes about (j / 32) * 16 + 5 * 8 per lane.
// Column j of segment s: hin[0..j] (shared memory, unrotated), hn = the
// subdiagonal entry (||w||); the rotated column goes to col[0..j] (shared
// memory, another array) and to R.  stop: the segment stops after this
// column whatever its residual (the last column of a cycle).
__device__ bool givens_core(const GivensArgs& ga, int s, int j, const double2* hin, double hn, double2* col,
                            bool stop = false) {
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
    const double2 h0 = hin[0];
    const int per = (j + 31) / 32;
    const int b = min(j, lane * per), e = min(j, b + per);
    // this lane's maps composed: (A, B) = M_{e-1} o ... o M_b
    double2 A = make_double2(1, 0), B = make_double2(0, 0);
    for (int i = b; i < e; ++i) {
        const double2 Ai = make_double2(-sn[i].x, sn[i].y);
        const double2 hi1 = hin[i + 1];
        const double2 Bi = make_double2(cs[i] * hi1.x, cs[i] * hi1.y);
        B = gv_fma(Ai, B, Bi);
        A = gv_mul(Ai, A);
    }
    // inclusive scan over the lanes: (A, B) <- (A, B) o (A, B) of lane - d
#pragma unroll 1
    for (int d = 1; d < 32; d <<= 1) {
        const double2 Ao = make_double2(__shfl_up_sync(0xffffffffu, A.x, d), __shfl_up_sync(0xffffffffu, A.y, d));
        const double2 Bo = make_double2(__shfl_up_sync(0xffffffffu, B.x, d), __shfl_up_sync(0xffffffffu, B.y, d));
        if (lane >= d) {
            B = gv_fma(A, Bo, B);
            A = gv_mul(A, Ao);
        }
    }
    // exclusive prefix: the composition of the lanes below
    double2 Ae = make_double2(__shfl_up_sync(0xffffffffu, A.x, 1), __shfl_up_sync(0xffffffffu, A.y, 1));
    double2 Be = make_double2(__shfl_up_sync(0xffffffffu, B.x, 1), __shfl_up_sync(0xffffffffu, B.y, 1));
    if (lane == 0) { Ae = make_double2(1, 0); Be = make_double2(0, 0); }
    double2 a = gv_fma(Ae, h0, Be);                 // a_b
    for (int i = b; i < e; ++i) {
        const double c = cs[i];
        const double2 si = sn[i];
        const double2 hi1 = hin[i + 1];
        col[i] = gv_fma(si, hi1, make_double2(c * a.x, c * a.y));
        a = gv_fma(make_double2(-si.x, si.y), a, make_double2(c * hi1.x, c * hi1.y));
    }
    // a_j: the carry out of the last non-empty range (h_0 when j = 0)
    const int last = j > 0 ? (j - 1) / per : 0;
    a = make_double2(__shfl_sync(0xffffffffu, a.x, last), __shfl_sync(0xffffffffu, a.y, last));
    if (j == 0) a = h0;
    // the new rotation, from (a_j, ||w||): c = |a| / d, s = (a / |a|) ||w|| / d, d = sqrt(|a|^2 + ||w||^2)
    const double n2a = a.x * a.x + a.y * a.y, d2 = n2a + hn * hn;
    double cj;
    double2 sj;
    if (d2 == 0.0) { cj = 1.0; sj = make_double2(0, 0); }
    else if (n2a == 0.0) { cj = 0.0; sj = make_double2(1.0, 0.0); }
    else {
        const double ia = rsqrt(n2a), id = rsqrt(d2);
        cj = n2a * ia * id;
        const double f = hn * ia * id;
        sj = make_double2(a.x * f, a.y * f);
    }
    int keep = 0;
    if (lane == 0) {
        ga.cs[(int64_t)s * m + j] = cj;
        ga.sn[(int64_t)s * m + j] = sj;
        col[j] = make_double2(cj * a.x + sj.x * hn, cj * a.y + sj.y * hn);
        double2* g = ga.gv + (int64_t)s * (m + 1);
        const double2 gj = g[j];
        const double2 gn = make_double2(-(sj.x * gj.x + sj.y * gj.y), -(sj.x * gj.y - sj.y * gj.x));   // -conj(s) g_j
        g[j + 1] = gn;
        g[j] = make_double2(cj * gj.x, cj * gj.y);
        if (ga.gmon && s == 0) *ga.gmon = gn;
        ga.kused[s] = j + 1;
        ga.beta[s] = hn;
        const double t = ga.target[s];
        keep = !(stop || gn.x * gn.x + gn.y * gn.y <= t * t || hn == 0.0);
        if (!keep) ga.active[s] = 0;
        else if (ga.nact) atomicAdd(ga.nact, 1);
    }
    __syncwarp();
    double2* out = ga.Rm + ((int64_t)s * m + j) * m;          // column j, rows 0..j
    for (int i = lane; i <= j; i += 32) out[i] = col[i];
    return __shfl_sync(0xffffffffu, keep, 0) != 0;
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
                gsh[i].x -= c[p].x * yq.x - c[p].y * yq.y;
                gsh[i].y -= c[p].x * yq.y + c[p].y * yq.x;
            }
        }
        for (int i = lane + 32 * NP; i < q; i += 32) {
            const double2 v = R[(int64_t)q * m + i];
            gsh[i].x -= v.x * yq.x - v.y * yq.y;
            gsh[i].y -= v.x * yq.y + v.y * yq.x;
        }
        __syncwarp();
    }
}

}  // namespace thm
