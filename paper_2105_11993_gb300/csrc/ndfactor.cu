// Numeric factorisation over the nested-dissection trees (nd.cuh): a
// multifrontal elimination in FP64, one launch per depth of the trees (over
// the nodes of all subdomains), deepest first.  A node's front is the dense
// (s+b)^2 matrix of its own entries plus its children's Schur complements;
//   W = F_ss^{-1} (Gauss-Jordan, partial pivoting inside the block, one Newton step),
//   H = W F_sb,   U = F_bb - F_bs H (the parent's share),
// and W, -H^T (forward rows) and -H (backward rows) go straight into the
// sliced layout the solve reads.  The same kernel factorises the complex
// T = P + iB (the full 2x2 block operator, 2-D: B diagonal).
//
// Pivoting stays inside a node, and that is not enough: a node's subtree is a
// cavity with conducting walls, and near one of its resonances S = F_ss is
// nearly singular though P is not.  H and U are then large and the digits of
// F_bb are lost in U.  Such a node shows in the entries of H, which are of
// order 1 elsewhere.  A node with |H| > ND_GROWTH names the unknowns that make
// it singular (nd_pick: one for each near-null direction of S), they move to
// the parent, the trees of these subdomains are built again and only they are
// factorised again, until no node is left.  Measured on 64 subdomains of 32x32
// order-2 cells with tile coefficients, 40 inputs, error of the FP64 solve
// against a refined one: without the moves up to 3.5 (5 inputs above 1e-9),
// with them at most 1.3e-11, for 0.02% more values.  4 subdomains of 32x32
// order-2 cells, uniform, 16 cells per wavelength: error 9e-4 -> 9e-15, and
// 2416 -> 509 Arnoldi steps of a mixed sweep.
// The bound: 1000 leaves errors of 6e-9 on the 40 inputs; 30 moves 3 times as
// many unknowns and factorises again more often (27 ms instead of 18 in the
// mean) for errors that are no smaller in the worst input (9e-12).
#include <algorithm>

#include "common.cuh"
#include "ndsolve.cuh"

namespace thm {

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Arithmetic of the two factor types.
template <class T> struct NdArith;
template <> struct NdArith<double> {
    static __device__ __forceinline__ double zero() { return 0.0; }
    static __device__ __forceinline__ double one() { return 1.0; }
    static __device__ __forceinline__ double mag(double a) { return fabs(a); }
    static __device__ __forceinline__ double size(double a) { return fabs(a); }      // mag within a factor of 1.5
    static __device__ __forceinline__ double inv(double a) { return 1.0 / a; }
    static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
    static __device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
    static __device__ __forceinline__ double neg(double a) { return -a; }
    static __device__ __forceinline__ double add(double a, double b) { return a + b; }
};
template <> struct NdArith<double2> {
    static __device__ __forceinline__ double2 zero() { return make_double2(0, 0); }
    static __device__ __forceinline__ double2 one() { return make_double2(1, 0); }
    static __device__ __forceinline__ double mag(double2 a) { return hypot(a.x, a.y); }
    static __device__ __forceinline__ double size(double2 a) { return fabs(a.x) + fabs(a.y); }
    static __device__ __forceinline__ double2 inv(double2 a) {
        const double d = a.x * a.x + a.y * a.y;
        return make_double2(a.x / d, -a.y / d);
    }
    static __device__ __forceinline__ double2 mul(double2 a, double2 b) { return zmul(a, b); }
    static __device__ __forceinline__ double2 fma_(double2 a, double2 b, double2 c) {
        return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
    }
    static __device__ __forceinline__ double2 neg(double2 a) { return make_double2(-a.x, -a.y); }
    static __device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
};

// Pivot of column k: the row of the largest |col[i * ld]|, k <= i < m (lowest
// index on ties), for the whole block; -1: it is zero, -2: not finite.
template <class T>
__device__ int nd_pivot(const T* col, int k, int m, int64_t ld) {
    using A = NdArith<T>;
    __shared__ double s_best[32];
    __shared__ int s_at[32];
    __shared__ int s_piv;
    const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double best = -1;
    int bi = -1;
    for (int i = k + tid; i < m; i += nt) {
        const double v = A::mag(col[(int64_t)i * ld]);
        if (v > best || !(v == v)) { best = v; bi = i; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (oi >= 0 && (bi < 0 || ov > best || (ov == best && oi < bi) || !(ov == ov))) { best = ov; bi = oi; }
    }
    if (lane == 0) { s_best[warp] = best; s_at[warp] = bi; }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < (nt >> 5); ++w)
            if (s_at[w] >= 0 && (bi < 0 || s_best[w] > best || (s_best[w] == best && s_at[w] < bi) || !(s_best[w] == s_best[w]))) {
                best = s_best[w];
                bi = s_at[w];
            }
        s_piv = (best > 0 && isfinite(best)) ? bi : best == 0 ? -1 : -2;
    }
    __syncthreads();
    return s_piv;
}

// Undoes the row interchanges of an inversion as column interchanges, last first.
template <class T>
__device__ void nd_unswap(T* W, int m, int ld, const int* perm) {
    for (int i = threadIdx.x; i < m; i += blockDim.x)
        for (int k = m - 1; k >= 0; --k) {
            const int p = perm[k];
            if (p != k) {
                const T a = W[(int64_t)i * ld + k];
                W[(int64_t)i * ld + k] = W[(int64_t)i * ld + p];
                W[(int64_t)i * ld + p] = a;
            }
        }
    __syncthreads();
}

// In-place inverse of the m x m block W (row stride ld) by Gauss-Jordan with
// partial pivoting, one CTA.  fcol, frow: m entries of shared memory each.
// 0, or on a zero pivot 1, on a non-finite one 2.
template <class T>
__device__ int nd_invert(T* W, int m, int ld, int* perm, T* fcol, T* frow) {
    using A = NdArith<T>;
    const int nt = blockDim.x, tid = threadIdx.x;
    const int di = nt / m, dj = nt % m, i0 = tid / m, j0 = tid % m;   // this thread's walk over the block
    for (int k = 0; k < m; ++k) {
        const int p = nd_pivot(W + k, k, m, ld);
        if (p < 0) return -p;
        if (tid == 0) perm[k] = p;
        // row k of the result (the pivot row over the pivot) and column k, staged
        const T ip = A::inv(W[(int64_t)p * ld + k]);
        for (int j = tid; j < m; j += nt) {
            frow[j] = j == k ? ip : A::mul(W[(int64_t)p * ld + j], ip);
            // rows k and p change places: row p takes the old row k
            const T c = W[(int64_t)(j == p ? k : j) * ld + k];
            fcol[j] = j == k ? A::zero() : A::neg(c);
        }
        __syncthreads();
        if (p != k)
            for (int j = tid; j < m; j += nt) W[(int64_t)p * ld + j] = W[(int64_t)k * ld + j];
        __syncthreads();
        for (int i = i0, j = j0; i < m;) {
            const int64_t o = (int64_t)i * ld + j;
            W[o] = i == k ? frow[j] : A::fma_(fcol[i], frow[j], j == k ? A::zero() : W[o]);
            i += di;
            j += dj;
            if (j >= m) { j -= m; ++i; }
        }
        __syncthreads();
    }
    nd_unswap(W, m, ld, perm);
    return 0;
}

// The same for blocks that outgrow shared memory, NB columns at a time: the
// panel of all m rows is eliminated in shared memory (columns contiguous), and
// then the other columns take its NB steps at once,
//     W_j = (W_j without the pivot rows) + X (pivot rows of W_j), X the panel,
// so W goes through L2 m / NB times instead of m times.  What bounds it then is
// the CTA's FP64 units (m^3 multiply-adds at 2 per clock).
template <class T, int NB>
__device__ __noinline__ int nd_invert_panels(T* W, int m, int ld, int* perm, T* X) {
    using A = NdArith<T>;
    __shared__ T s_row[NB];
    const int nt = blockDim.x, tid = threadIdx.x;
    // a column per thread, its rows shared out where there are fewer columns than threads
    const int cw = min(nt, (m + 31) / 32 * 32), ng = nt / cw, grp = tid / cw, tc = tid - grp * cw;
    for (int k0 = 0; k0 < m; k0 += NB) {
        const int nb = min(NB, m - k0);
        for (int t = tid; t < m * nb; t += nt) {
            const int i = t / nb, q = t - i * nb;
            X[q * m + i] = W[(int64_t)i * ld + k0 + q];
        }
        __syncthreads();
        for (int q = 0; q < nb; ++q) {
            const int k = k0 + q, p = nd_pivot(X + q * m, k, m, 1);
            if (p < 0) return -p;
            if (tid == 0) perm[k] = p;
            const T ip = A::inv(X[q * m + p]);
            if (tid < nb) s_row[tid] = tid == q ? ip : A::mul(X[tid * m + p], ip);
            __syncthreads();
            if (p != k && tid < nb) X[tid * m + p] = X[tid * m + k];
            __syncthreads();
            for (int i = tid; i < m; i += nt) {
                const T f = A::neg(X[q * m + i]);
                for (int c = 0; c < nb; ++c)
                    X[c * m + i] = i == k ? s_row[c] : A::fma_(f, s_row[c], c == q ? A::zero() : X[c * m + i]);
            }
            __syncthreads();
        }
        for (int c0 = 0; c0 < m; c0 += cw) {
            const int j = c0 + tc;
            const bool on = grp < ng && j < m && (j < k0 || j >= k0 + nb);
            if (on && grp == 0)
                for (int q = 0; q < nb; ++q) {
                    const int p = perm[k0 + q];
                    if (p == k0 + q) continue;
                    const T a = W[(int64_t)(k0 + q) * ld + j];
                    W[(int64_t)(k0 + q) * ld + j] = W[(int64_t)p * ld + j];
                    W[(int64_t)p * ld + j] = a;
                }
            __syncthreads();
            T t[NB];
#pragma unroll
            for (int q = 0; q < NB; ++q) t[q] = on && q < nb ? W[(int64_t)(k0 + q) * ld + j] : A::zero();
            __syncthreads();
            constexpr int U = 4;                       // rows in flight
            if (on)
                for (int i0 = grp * U; i0 < m; i0 += ng * U) {
                    T v[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int i = i0 + u;
                        v[u] = i < m && (i < k0 || i >= k0 + nb) ? W[(int64_t)i * ld + j] : A::zero();
                    }
#pragma unroll
                    for (int q = 0; q < NB; ++q)
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (q < nb) v[u] = A::fma_(X[q * m + min(i0 + u, m - 1)], t[q], v[u]);
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (i0 + u < m) W[(int64_t)(i0 + u) * ld + j] = v[u];
                }
        }
        __syncthreads();
        for (int t = tid; t < m * nb; t += nt) {
            const int i = t / nb, q = t - i * nb;
            W[(int64_t)i * ld + k0 + q] = X[q * m + i];
        }
        __syncthreads();
    }
    nd_unswap(W, m, ld, perm);
    return 0;
}

// Largest over the block's threads (NaN if there is one); red: 32 entries.
__device__ __forceinline__ double nd_block_max(double v, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double u = __shfl_xor_sync(0xffffffffu, v, o);
        if (u > v || u != u) v = u;
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
        if (red[w] > v || red[w] != red[w]) v = red[w];
    return v;
}

// Entries of H above this move unknowns to the parent.
constexpr double ND_GROWTH = 100;

// What a factorisation reports: status[0] a non-finite pivot, [1] the number of
// entries of moves: {node, local row} (at most one per local row) for an
// unknown that moves up, {node, -1} for a node with a zero pivot.
struct NdReport {
    int* status;
    int2* moves;
    __device__ void add(int node, int row) const { moves[atomicAdd(&status[1], 1)] = make_int2(node, row); }
};

// The unknowns of a node that must not be eliminated there.  G = [W | H], s x
// (s + b): taking unknown d out of the block is a principal pivot step on G,
//     G_ij -= G_id G_dj / G_dd   (i, j != d),   G_id = -G_id / G_dd,
// after which column d belongs to the H of the rows that stay.  W is about
// sum_k v_k v_k^T / lambda_k over the near-null directions of S, so the
// largest diagonal entry is an unknown with a large part in one of them; they
// go one by one until the H of the rest is below ND_GROWTH.  gone, col: s entries each.
template <class T>
__device__ __noinline__ void nd_pick(T* G, int s, int b, int ld, T* col, int* gone, const int32_t* rows, int node, NdReport rep) {
    using A = NdArith<T>;
    __shared__ double s_red[32], s_val[32];
    __shared__ int s_idx[32];
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < s; i += nt) gone[i] = 0;
    __syncthreads();
    for (int left = s; left > 0; --left) {
        double best = -1;
        int d = -1;
        for (int i = tid; i < s; i += nt) {
            const double v = gone[i] ? -1.0 : A::mag(G[(int64_t)i * ld + i]);
            if (v > best) { best = v; d = i; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ov = __shfl_xor_sync(0xffffffffu, best, o);
            const int od = __shfl_xor_sync(0xffffffffu, d, o);
            if (od >= 0 && (d < 0 || ov > best || (ov == best && od < d))) { best = ov; d = od; }
        }
        __syncthreads();
        if (lane == 0) { s_val[warp] = best; s_idx[warp] = d; }
        __syncthreads();
        best = s_val[0];
        d = s_idx[0];
        for (int w = 1; w < (nt >> 5); ++w)
            if (s_idx[w] >= 0 && (d < 0 || s_val[w] > best || (s_val[w] == best && s_idx[w] < d))) { best = s_val[w]; d = s_idx[w]; }
        if (d < 0 || !(best > 0)) {            // (not reached from finite entries but for a zero diagonal) all of them go
            for (int i = tid; i < s; i += nt)
                if (!gone[i]) rep.add(node, rows[i]);
            return;
        }
        const T id = A::inv(G[(int64_t)d * ld + d]);
        for (int i = tid; i < s; i += nt) col[i] = A::neg(A::mul(G[(int64_t)i * ld + d], id));
        __syncthreads();
        if (tid == 0) {
            gone[d] = 1;
            rep.add(node, rows[d]);
        }
        __syncthreads();
        double hm = 0;
        for (int t = tid; t < s * (s + b); t += nt) {
            const int i = t / (s + b), j = t - i * (s + b);
            if (gone[i]) continue;
            T* g = G + (int64_t)i * ld + j;
            const T v = j == d ? col[i] : A::fma_(col[i], G[(int64_t)d * ld + j], *g);
            *g = v;
            if (j >= s || gone[j]) {
                const double a = A::size(v);
                if (!(a <= hm)) hm = a;
            }
        }
        if (nd_block_max(hm, s_red) <= ND_GROWTH) return;
    }
}

__device__ __forceinline__ int nd_find(const int32_t* a, int n, int32_t v) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo < n && a[lo] == v ? lo : -1;
}

// Entry (row, column) of the rows of a level in the factor.
__device__ __forceinline__ int64_t nd_at(const int2* slt, int row, int col) {
    return (int64_t)slt[row >> 5].x * 128 + (col >> 2) * 128 + (row & 31) * 4 + (col & 3);
}

// out(i, j, init(i, j) + sum_k A[i][k] col(j)[at(k)]) for an m x n product, one
// CTA, the sums in the order of k.  Large products take 8 rows at a time per thread:
// one element of B serves 8 multiply-adds, and those of A are the same for a
// warp.  (One at a time every multiply-add waits for two loads: with the whole
// product from L2, and the inverse a column at a time, the factorisation of 8
// subdomains of 16^3 cells, whose roots have some 1,500 unknowns, took 7.1 s
// instead of 3.1, of 64 such 2.6 s instead of 1.1.)
template <class T, bool BIG, class Init, class Col, class At, class Out>
__device__ __forceinline__ void nd_product(int m, int n, int kk, const T* A, int lda, Init init, Col col, At at, Out out) {
    using Ar = NdArith<T>;
    constexpr int RB = 8;
    if (BIG && m * n >= 2 * RB * (int)blockDim.x) {
        const int mb = (m + RB - 1) / RB;
        for (int t = threadIdx.x; t < mb * n; t += blockDim.x) {
            const int ib = t / n, j = t - ib * n, i0 = ib * RB;
            const T* bj = col(j);
            const T* a[RB];
            T c[RB];
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                a[r] = A + (int64_t)min(i0 + r, m - 1) * lda;
                c[r] = init(min(i0 + r, m - 1), j);
            }
            for (int k = 0; k < kk; ++k) {
                const T b = bj[at(k)];
#pragma unroll
                for (int r = 0; r < RB; ++r) c[r] = Ar::fma_(a[r][k], b, c[r]);
            }
#pragma unroll
            for (int r = 0; r < RB; ++r)
                if (i0 + r < m) out(i0 + r, j, c[r]);
        }
        return;
    }
    for (int t = threadIdx.x; t < m * n; t += blockDim.x) {
        const int i = t / n, j = t - i * n;
        const T *a = A + (int64_t)i * lda, *bj = col(j);
        T c = init(i, j);
        for (int k = 0; k < kk; ++k) c = Ar::fma_(a[k], bj[at(k)], c);
        out(i, j, c);
    }
}

template <class T, bool BIG, class Out>
__device__ __forceinline__ void nd_gemm(int m, int n, int kk, const T* A, int lda, const T* B, int ldb, Out out) {
    nd_product<T, BIG>(m, n, kk, A, lda, [](int, int) { return NdArith<T>::zero(); },
                       [&](int j) { return B + j; }, [&](int k) { return (int64_t)k * ldb; }, out);
}

// One CTA per node of a depth.  BIG: blocks of the depth outgrow shared memory
// (more than 160 unknowns, 113 complex); they are inverted in place in the
// front, `panel` columns at a time (0: one), and products take 8 rows at a time.
// (A kernel of its own: its registers would halve the CTAs per SM of the many
// small nodes.)
template <class T, bool BIG>
__global__ void __launch_bounds__(512) k_nd_factor(NdTables tab, const NdNode* __restrict__ nodes, int64_t node0, const int32_t* __restrict__ rows,
                            const int32_t* __restrict__ cmap, const int32_t* __restrict__ childs, int C, int panel,
                            int max_s, const int64_t* __restrict__ slice_ptr, const int32_t* __restrict__ col,
                            const uint8_t* __restrict__ pad, const double* __restrict__ val,
                            const double* __restrict__ bg, const double* __restrict__ bs, T* front, const T* below,
                            T* aux, T* fac, NdReport rep) {
    using A = NdArith<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* fcol = reinterpret_cast<T*>(smem_raw);
    T* frow = fcol + max_s;
    T* blk = frow + max_s;
    int* perm = reinterpret_cast<int*>(blk + (size_t)max_s * (BIG ? panel : max_s));
    const NdNode N = nodes[node0 + blockIdx.x];
    const int s = N.s, b = N.b, n = s + b, tid = threadIdx.x, nt = blockDim.x;
    const int32_t* rs = rows + N.rows0;
    T* F = front + N.front;
    for (int t = tid; t < n * n; t += nt) F[t] = A::zero();
    __syncthreads();
    // the node's own entries: rows of its unknowns, columns among them and the ancestors'
    for (int i = tid; i < s; i += nt) {
        const int64_t r = rs[i];
        const int64_t sl = r / SELL_C;
        const int64_t base = slice_ptr[sl] + (r % SELL_C);
        const int w = (int)((slice_ptr[sl + 1] - slice_ptr[sl]) / SELL_C);
        for (int q = 0; q < w; ++q) {
            const int64_t idx = base + (int64_t)q * SELL_C;
            if (pad[idx]) continue;
            const int32_t c = col[idx];
            int j = nd_find(rs, s, c);
            const bool anc = j < 0;
            if (anc) {
                j = nd_find(rs + s, b, c);
                if (j < 0) continue;                  // eliminated below: in that node's front
                j += s;
            }
            T v = A::zero();
            if constexpr (NdCplx<T>::value) v.x = val[idx]; else v = val[idx];
            F[(int64_t)i * n + j] = v;
            if (anc) F[(int64_t)j * n + i] = v;
        }
        if constexpr (NdCplx<T>::value) F[(int64_t)i * n + i].y = bg[r] + bs[r];
    }
    __syncthreads();
    for (int k = 0; k < N.nchild; ++k) {
        const NdNode K = nodes[childs[N.child0 + k]];
        const T* G = below + K.front;
        const int kn = K.s + K.b;
        const int32_t* cm = cmap + K.cmap0;
        for (int t = tid; t < K.b * K.b; t += nt) {
            const int i = t / K.b, j = t - i * K.b;
            T* d = F + (int64_t)cm[i] * n + cm[j];
            *d = A::add(*d, G[(int64_t)(K.s + i) * kn + K.s + j]);
        }
        __syncthreads();
    }
    if (s == 0) return;
    // scratch of the node: S (when it is inverted in place), a residual, a product
    T* X = aux + 3 * N.front;
    T* Rs = X + (int64_t)n * n;
    T* Y = Rs + (int64_t)n * n;
    T* W = F;
    const T* S = F;
    int ld = n;
    if (!BIG) {
        W = blk;
        ld = s;
        for (int t = tid; t < s * s; t += nt) W[t] = F[(int64_t)(t / s) * n + t % s];
    } else {
        for (int t = tid; t < s * s; t += nt) X[(int64_t)(t / s) * n + t % s] = F[(int64_t)(t / s) * n + t % s];
        S = X;
    }
    __syncthreads();
    int bad;
    if constexpr (BIG)
        bad = panel == 16  ? nd_invert_panels<T, 16>(W, s, ld, perm, blk)
              : panel == 8 ? nd_invert_panels<T, 8>(W, s, ld, perm, blk)
                           : nd_invert(W, s, ld, perm, fcol, frow);
    else
        bad = nd_invert(W, s, ld, perm, fcol, frow);
    if (bad) {
        const int node = (int)(node0 + blockIdx.x);
        if (tid == 0 && bad == 2) atomicExch(&rep.status[0], 1);
        if (tid == 0 && bad == 1) rep.add(node, -1);
        if (bad == 1 && b > 0)                         // exactly singular: all of it moves up
            for (int i = tid; i < s; i += nt) rep.add(node, rs[i]);
        return;
    }
    // One Newton step, W += W (I - S W): Gauss-Jordan leaves an error of
    // u cond(S)^2 or so in W, and the Schur complements of the parents inherit
    // it (measured on 32x32 order-1 cells at omega = 4: the solve's error is
    // 6e-13 without this and the one of H below, 1.4e-14 with them).
    nd_gemm<T, BIG>(s, s, s, S, n, W, ld, [&](int i, int j, T a) { Rs[(int64_t)i * n + j] = A::add(i == j ? A::one() : A::zero(), A::neg(a)); });
    __syncthreads();
    nd_gemm<T, BIG>(s, s, s, W, ld, Rs, n, [&](int i, int j, T a) { Y[(int64_t)i * n + j] = A::add(W[(int64_t)i * ld + j], a); });
    __syncthreads();
    for (int t = tid; t < s * s; t += nt) W[(int64_t)(t / s) * ld + t % s] = Y[(int64_t)(t / s) * n + t % s];
    __syncthreads();
    if (N.root_rows > 0) {                             // the root: its rows are shared out over the CTAs
        for (int t = tid; t < s * s; t += nt) {
            const int i = t / s, j = t - i * s, rk = i / N.root_rows;
            const NdPart P = tab.parts[(int64_t)N.sub * C + rk];
            const NdLev L = tab.levs[P.lev0 + P.nlev];
            fac[nd_at(tab.slt + P.slt0 + L.sltf, i - rk * N.root_rows, j)] = W[(int64_t)i * ld + j];
        }
        return;
    }
    const int2* sf = tab.slt + N.slt_f;
    for (int t = tid; t < s * s; t += nt) {
        const int i = t / s, j = t - i * s;
        fac[nd_at(sf, N.row_f + i, j)] = W[(int64_t)i * ld + j];
    }
    if (b == 0) return;
    const int2* sb = tab.slt + N.slt_b;
    // H = W F_sb with a residual correction H += W (F_sb - S H)
    const T* Fb = F + s;
    nd_gemm<T, BIG>(s, b, s, W, ld, Fb, n, [&](int i, int j, T a) { Y[(int64_t)i * n + j] = a; });
    __syncthreads();
    nd_gemm<T, BIG>(s, b, s, S, n, Y, n, [&](int i, int j, T a) { Rs[(int64_t)i * n + j] = A::add(Fb[(int64_t)i * n + j], A::neg(a)); });
    __syncthreads();
    double hm = 0;
    nd_gemm<T, BIG>(s, b, s, W, ld, Rs, n, [&](int i, int j, T a) {
        const T h = A::neg(A::add(Y[(int64_t)i * n + j], a));
        const double v = A::size(h);
        if (!(v <= hm)) hm = v;
        fac[nd_at(sf, N.row_f + s + j, i)] = h;
        fac[nd_at(sb, N.row_b + i, j)] = h;
    });
    __syncthreads();
    T* U = F + (int64_t)s * n + s;
    nd_product<T, BIG>(b, b, s, F + (int64_t)s * n, n, [&](int i, int j) { return U[(int64_t)i * n + j]; },
                       [&](int j) { return fac + nd_at(sf, N.row_f + s + j, 0); }, [](int k) { return (k >> 2) * 128 + (k & 3); },
                       [&](int i, int j, T a) { U[(int64_t)i * n + j] = a; });
    __shared__ double s_red[32];
    hm = nd_block_max(hm, s_red);
    if (hm <= ND_GROWTH) return;
    if (!isfinite(hm)) {
        if (tid == 0) atomicExch(&rep.status[0], 1);
        return;
    }
    for (int t = tid; t < s * n; t += nt) {            // [W | H] over the scratch, which is free
        const int i = t / n, j = t - i * n;
        Y[t] = j < s ? W[(int64_t)i * ld + j] : A::neg(fac[nd_at(sb, N.row_b + i, j - s)]);
    }
    __syncthreads();
    nd_pick<T>(Y, s, b, n, fcol, perm, rs, (int)(node0 + blockIdx.x), rep);
}

NdTables nd_tables(const thm_sys* s, bool cplx) {
    const auto& own = cplx ? s->ownc : s->own;
    const NdDev& D = own ? own->d : s->m->ndd;
    NdTables T{};
    T.parts = D.parts.p; T.levs = D.levs.p; T.slt = D.slt.p;
    T.rowd = D.rowd.p; T.rowm = D.rowm.p; T.ymap = D.ymap.p; T.rmap = D.rmap.p;
    T.idx = D.idx.p; T.perm = D.perm.p; T.welem = D.welem.p; T.subs = s->m->d_subs.p;
    T.mw = s->m->nd.mw;
    return T;
}

void require_nd(const thm_mesh* m) {
    THM_REQUIRE(m->nd_ok, "subdomain too large for the shared-memory block solve");
}

// dst = base, `add` behind it, and room for `more` entries
template <class X>
static void append(DArr<X>& dst, const DArr<X>& base, const std::vector<X>& add, cudaStream_t st, size_t more = 0) {
    DArr<X> a;
    a.alloc(base.n + add.size() + more);
    if (base.n) THM_CUDA(cudaMemcpyAsync(a.p, base.p, base.n * sizeof(X), cudaMemcpyDeviceToDevice, st));
    if (!add.empty()) THM_CUDA(cudaMemcpyAsync(a.p + base.n, add.data(), add.size() * sizeof(X), cudaMemcpyHostToDevice, st));
    if (&dst == &base) THM_CUDA(cudaStreamSynchronize(st));      // its array goes now
    std::swap(dst.p, a.p);
    std::swap(dst.n, a.n);
}

// A subdomain whose moves make its factor this many times larger keeps the one
// it has: moves are for a few unknowns of a few nodes (1.0005 times the values
// at most on the inputs above, 1.06 on uniform media), and coefficients or
// cells that show large H everywhere would fill the tree up to one dense block.
constexpr double ND_FILL = 2;
constexpr size_t ND_FACTOR_SMEM = 225 * 1024;      // dynamic, beside 1 KB or so of static shared memory
constexpr int ND_PASSES = 12;               // (2 or 3 are the rule)

// Builds the trees of the subdomains of `found` again with these unknowns of
// nodes of H in the parents, and puts their tables behind the present ones
// (own: null while these are the mesh's).  False, and no tables changed: there
// is nothing left to move, or the tables outgrow the solve kernel.
// kept [n_sub]: subdomains that are left as they are, more of which are found
// here; singular: a zero pivot is in one of these.
static bool move_up(const thm_sys* s, const NdHost& H, const std::vector<int2>& found, std::vector<char>& kept, bool& singular,
                    std::unique_ptr<NdOwn>& own, NdHost& out) {
    const thm_mesh* m = s->m;
    cudaStream_t st = s->st;
    const int C = m->nd.C;
    const auto before = own ? own->moves : std::vector<std::vector<NdMove>>(m->n_sub);
    auto moves = before;
    std::vector<char> zero(m->n_sub, 0);
    std::vector<int> list;
    for (const int2& f : found) {
        const NdRef& r = H.node_ref[f.x];
        if (f.y < 0) zero[r.sub] = 1;
        if (f.y < 0 || kept[r.sub]) continue;
        auto& v = moves[r.sub];
        auto it = std::lower_bound(v.begin(), v.end(), f.y, [](const NdMove& a, int row) { return a.row < row; });
        if (it != v.end() && it->row == f.y) it->node = r.parent;
        else v.insert(it, NdMove{f.y, r.parent});
        list.push_back(r.sub);
    }
    std::sort(list.begin(), list.end());
    list.erase(std::unique(list.begin(), list.end()), list.end());
    int p = 0;
    while ((1 << p) < C) ++p;
    while (true) {
        const bool ok = !list.empty() && build_tables(m, out, list, p, &moves);
        // those that stay within ND_FILL, or (tables too large) all but the one with the most moves
        auto most = std::max_element(list.begin(), list.end(), [&](int a, int b) { return moves[a].size() < moves[b].size(); });
        std::vector<int> fit;
        for (size_t i = 0; i < list.size(); ++i)
            if (ok ? out.welem[i] <= ND_FILL * m->nd.welem[list[i]] : list[i] != *most) fit.push_back(list[i]);
        if (ok && fit.size() == list.size()) break;
        for (int q : list)
            if (!std::binary_search(fit.begin(), fit.end(), q)) {
                kept[q] = 1;
                moves[q] = before[q];
            }
        list.swap(fit);
        if (list.empty()) break;
    }
    for (int q = 0; q < m->n_sub; ++q)
        singular = singular || (zero[q] && !std::binary_search(list.begin(), list.end(), q));
    if (list.empty()) return false;
    const NdDev& B = own ? own->d : m->ndd;
    const int64_t fac0 = own ? own->fac_elems : m->nd.fac_elems;
    if (!place_tables(out, NdPlace{B.levs.n, B.slt.n, B.rowd.n, B.ymap.n, B.rmap.n, B.idx.n, B.perm.n, (size_t)fac0})) {
        singular = std::any_of(zero.begin(), zero.end(), [](char z) { return z != 0; });
        return false;
    }
    std::unique_ptr<NdOwn> o(new NdOwn());
    append(o->d.levs, B.levs, out.levs, st);
    append(o->d.slt, B.slt, out.slt, st);
    append(o->d.rowd, B.rowd, out.rowd, st);
    append(o->d.rowm, B.rowm, out.rowm, st);
    append(o->d.ymap, B.ymap, out.ymap, st);
    append(o->d.rmap, B.rmap, out.rmap, st);
    append(o->d.idx, B.idx, out.idx, st);
    append(o->d.perm, B.perm, out.perm, st);
    o->parts = own ? own->parts : m->nd.parts;
    o->welem = own ? own->welem : m->nd.welem;
    for (size_t i = 0; i < list.size(); ++i) {
        for (int k = 0; k < C; ++k) o->parts[(size_t)list[i] * C + k] = out.parts[i * C + k];
        o->welem[list[i]] = out.welem[i];
    }
    o->d.parts.upload(o->parts, st);
    o->d.welem.upload(o->welem, st);
    o->d.nodes.upload(out.nodes, st);
    o->d.rows.upload(out.rows, st);
    o->d.cmap.upload(out.cmap, st);
    o->d.childs.upload(out.childs, st);
    o->z = larger(s->nd_sizes(&own == &s->ownc), out.z);
    o->fac_elems = fac0 + out.fac_elems;
    o->moves.swap(moves);
    THM_CUDA(cudaStreamSynchronize(st));               // the copies are done with both
    own.swap(o);
    return true;
}

template <class T>
static void factor(thm_sys* s, DArr<T>& fac, const char* what) {
    constexpr bool cplx = NdCplx<T>::value;
    const thm_mesh* m = s->m;
    cudaStream_t st = s->st;
    require_nd(m);
    std::unique_ptr<NdOwn>& own = cplx ? s->ownc : s->own;
    own.reset();
    fac.alloc(m->nd.fac_elems);
    fac.zero(st);
    DArr<T> front[2], aux;
    DArr<int> status;
    status.alloc(2);
    DArr<int2> moves;
    moves.alloc(m->n_loc + m->nd.nodes.size());
    std::vector<char> kept(m->n_sub, 0);
    THM_CUDA(cudaFuncSetAttribute(k_nd_factor<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ND_FACTOR_SMEM));
    THM_CUDA(cudaFuncSetAttribute(k_nd_factor<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ND_FACTOR_SMEM));
    NdHost again;                                      // the subdomains that are factorised again
    for (int passes = 0;; ++passes) {
        const bool first = passes == 0;
        const NdHost& H = first ? m->nd : again;
        const NdDev& D = first ? m->ndd : own->d;
        int64_t most[2] = {0, 0};
        const int nd = (int)H.depth_front.size();
        for (int d = 0; d < nd; ++d) most[d & 1] = std::max(most[d & 1], H.depth_front[d]);
        for (int k = 0; k < 2; ++k)
            if ((int64_t)front[k].n < most[k]) front[k].alloc(most[k]);
        if ((int64_t)aux.n < 3 * std::max(most[0], most[1])) aux.alloc(3 * std::max(most[0], most[1]));
        status.zero(st);
        for (int d = 0; d < nd; ++d) {
            const int64_t n0 = H.depth_node[d], cnt = H.depth_node[d + 1] - n0;
            const int ms = std::max(1, H.depth_s[d]), mn = H.depth_n[d];
            const bool big = (size_t)ms * ms * sizeof(T) > 200 * 1024;
            const size_t rest = (size_t)2 * ms * sizeof(T) + (size_t)ms * sizeof(int);
            int panel = 0;
            for (int w : {16, 8})                  // (8: more than 1,556 unknowns, 789 complex; 0: more than 2,742, 1,404)
                if (big && panel == 0 && rest + (size_t)ms * w * sizeof(T) <= ND_FACTOR_SMEM) panel = w;
            const size_t smem = rest + (size_t)ms * (big ? panel : ms) * sizeof(T);
            int threads = 32;
            while (threads < 512 && threads * 16 < mn * mn) threads *= 2;
            const auto kernel = big ? k_nd_factor<T, true> : k_nd_factor<T, false>;
            THM_LAUNCH(THM_K_SETUP, st, kernel<<<(unsigned)cnt, threads, smem, st>>>(
                nd_tables(s, cplx), D.nodes.p, n0, D.rows.p, D.cmap.p, D.childs.p, H.C, panel, ms,
                m->d_slice_ptr.p, m->d_sell_col.p, m->d_sell_pad.p, s->val64.p, s->bg64.p, s->bs64.p, front[d & 1].p,
                front[(d + 1) & 1].p, aux.p, fac.p, NdReport{status.p, moves.p}));
            THM_CUDA(cudaGetLastError());
        }
        std::vector<int> hs;
        status.download(hs, st);
        if (hs[0] != 0) fail(THM_ESINGULAR, what);
        if (hs[1] == 0) break;
        std::vector<int2> found(hs[1]);
        THM_CUDA(cudaMemcpyAsync(found.data(), moves.p, found.size() * sizeof(int2), cudaMemcpyDeviceToHost, st));
        THM_CUDA(cudaStreamSynchronize(st));
        std::sort(found.begin(), found.end(), [](const int2& a, const int2& b) { return a.x != b.x ? a.x < b.x : a.y < b.y; });
        NdHost next;
        if (passes == ND_PASSES) kept.assign(m->n_sub, 1);
        bool singular = false;
        const bool moved = move_up(s, H, found, kept, singular, own, next);
        if (singular) fail(THM_ESINGULAR, what);
        if (!moved) break;
        std::swap(again, next);
        const size_t n0 = fac.n;
        append(fac, fac, std::vector<T>(), st, again.fac_elems);
        THM_CUDA(cudaMemsetAsync(fac.p + n0, 0, (fac.n - n0) * sizeof(T), st));
    }
}

__global__ void k_to_float2(int64_t n, const double2* __restrict__ a, float2* __restrict__ b) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = make_float2((float)a[i].x, (float)a[i].y);
}
__global__ void k_to_float(int64_t n, const double* __restrict__ a, float* __restrict__ b) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = (float)a[i];
}

// The full-block factors (complex), FP64 and for the mixed mode FP32.
void ensure_factor_full(thm_sys* s, bool fp32) {
    THM_REQUIRE(s->m->dim == 2, "the full 2x2 block preconditioner is built for 2-D meshes (diagonal B) only");
    if (!s->facc64_ok) {
        factor<double2>(s, s->facc64, "a diagonal block of the complex subdomain operator T_i is singular");
        s->facc64_ok = true;
    }
    if (fp32 && !s->facc32_ok) {
        s->facc32.alloc(s->facc64.n);
        THM_LAUNCH(THM_K_SETUP, s->st, k_to_float2<<<(unsigned)((s->facc64.n + 255) / 256), 256, 0, s->st>>>(
            (int64_t)s->facc64.n, s->facc64.p, s->facc32.p));
        THM_CUDA(cudaGetLastError());
        s->facc32_ok = true;
    }
}

// The factorisation runs in FP64 for both modes (pivots and Schur updates in
// FP64); the mixed mode stores the factor rounded to FP32.
void ensure_factor(thm_sys* s, bool fp32) {
    if (!s->fac64_ok) {
        factor<double>(s, s->fac64, "a diagonal block of P_i = A_i - omega^2 M_i is singular "
                                    "(omega^2 is a natural-boundary eigenvalue of a subdomain block)");
        s->fac64_ok = true;
    }
    if (fp32 && !s->fac32_ok) {
        s->fac32.alloc(s->fac64.n);
        THM_LAUNCH(THM_K_SETUP, s->st, k_to_float<<<(unsigned)((s->fac64.n + 255) / 256), 256, 0, s->st>>>((int64_t)s->fac64.n, s->fac64.p, s->fac32.p));
        THM_CUDA(cudaGetLastError());
        s->fac32_ok = true;
    }
}

}  // namespace thm
