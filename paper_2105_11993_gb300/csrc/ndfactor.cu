// Numeric factorisation over the nested-dissection trees (nd.cuh): a
// multifrontal elimination in FP64, one launch per depth of the trees (over
// the nodes of all subdomains), deepest first.  A node's front is the dense
// (s+b)^2 matrix of its own entries plus its children's Schur complements;
//   W = F_ss^{-1} (Gauss-Jordan, partial pivoting inside the block, one Newton step),
//   H = W F_sb,   U = F_bb - F_bs H (the parent's share),
// and W, -H^T (forward rows) and -H (backward rows) go straight into the
// sliced layout the solve reads.  The same kernel factorises the complex
// T = P + iB (the full 2x2 block operator, 2-D: B diagonal).
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

// In-place inverse of the m x m block W (row stride ld) by Gauss-Jordan with
// partial pivoting, one CTA.  fcol, frow: m entries of shared memory each.
// False on a zero or non-finite pivot.
template <class T>
__device__ bool nd_invert(T* W, int m, int ld, int* perm, T* fcol, T* frow) {
    using A = NdArith<T>;
    __shared__ double s_best[32];
    __shared__ int s_at[32];
    __shared__ int s_piv;
    const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int di = nt / m, dj = nt % m, i0 = tid / m, j0 = tid % m;   // this thread's walk over the block
    for (int k = 0; k < m; ++k) {
        // pivot: largest |W[i][k]|, i >= k (lowest index on ties)
        double best = -1;
        int bi = -1;
        for (int i = k + tid; i < m; i += nt) {
            const double v = A::mag(W[(int64_t)i * ld + k]);
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
            perm[k] = bi;
            s_piv = (best > 0 && isfinite(best)) ? bi : -1;
        }
        __syncthreads();
        const int p = s_piv;
        if (p < 0) return false;
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
    // undo the row interchanges as column interchanges, last first
    for (int i = tid; i < m; i += nt)
        for (int k = m - 1; k >= 0; --k) {
            const int p = perm[k];
            if (p != k) {
                const T a = W[(int64_t)i * ld + k];
                W[(int64_t)i * ld + k] = W[(int64_t)i * ld + p];
                W[(int64_t)i * ld + p] = a;
            }
        }
    __syncthreads();
    return true;
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

// out(i, j, sum_k A[i][k] B[k][j]) for an m x n product, one CTA
template <class T, class Out>
__device__ __forceinline__ void nd_gemm(int m, int n, int kk, const T* A, int lda, const T* B, int ldb, Out out) {
    using Ar = NdArith<T>;
    for (int t = threadIdx.x; t < m * n; t += blockDim.x) {
        const int i = t / n, j = t - i * n;
        const T* a = A + (int64_t)i * lda;
        const T* b = B + j;
        T c = Ar::zero();
        for (int k = 0; k < kk; ++k) c = Ar::fma_(a[k], b[(int64_t)k * ldb], c);
        out(i, j, c);
    }
}

// One CTA per node of a depth.  smem_s: blocks of at most that many unknowns
// are inverted in shared memory, larger ones in place in the front.
template <class T>
__global__ void k_nd_factor(NdTables tab, const NdNode* __restrict__ nodes, int64_t node0, const int32_t* __restrict__ rows,
                            const int32_t* __restrict__ cmap, const int32_t* __restrict__ childs, int C, int smem_s,
                            int max_s, const int64_t* __restrict__ slice_ptr, const int32_t* __restrict__ col,
                            const uint8_t* __restrict__ pad, const double* __restrict__ val,
                            const double* __restrict__ bg, const double* __restrict__ bs, T* front, const T* below,
                            T* aux, T* fac, int* __restrict__ status) {
    using A = NdArith<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* fcol = reinterpret_cast<T*>(smem_raw);
    T* frow = fcol + max_s;
    T* blk = frow + max_s;
    int* perm = reinterpret_cast<int*>(blk + (smem_s > 0 ? (size_t)smem_s * smem_s : 0));
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
    if (s <= smem_s) {
        W = blk;
        ld = s;
        for (int t = tid; t < s * s; t += nt) W[t] = F[(int64_t)(t / s) * n + t % s];
    } else {
        for (int t = tid; t < s * s; t += nt) X[(int64_t)(t / s) * n + t % s] = F[(int64_t)(t / s) * n + t % s];
        S = X;
    }
    __syncthreads();
    if (!nd_invert(W, s, ld, perm, fcol, frow)) {
        if (tid == 0) atomicExch(status, 1);
        return;
    }
    // One Newton step, W += W (I - S W): Gauss-Jordan leaves an error of
    // u cond(S)^2 or so in W, and the Schur complements of the parents inherit
    // it (measured on 32x32 order-1 cells at omega = 4: the solve's error is
    // 6e-13 without this and the one of H below, 1.4e-14 with them).
    nd_gemm<T>(s, s, s, S, n, W, ld, [&](int i, int j, T a) { Rs[(int64_t)i * n + j] = A::add(i == j ? A::one() : A::zero(), A::neg(a)); });
    __syncthreads();
    nd_gemm<T>(s, s, s, W, ld, Rs, n, [&](int i, int j, T a) { Y[(int64_t)i * n + j] = A::add(W[(int64_t)i * ld + j], a); });
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
    nd_gemm<T>(s, b, s, W, ld, Fb, n, [&](int i, int j, T a) { Y[(int64_t)i * n + j] = a; });
    __syncthreads();
    nd_gemm<T>(s, b, s, S, n, Y, n, [&](int i, int j, T a) { Rs[(int64_t)i * n + j] = A::add(Fb[(int64_t)i * n + j], A::neg(a)); });
    __syncthreads();
    nd_gemm<T>(s, b, s, W, ld, Rs, n, [&](int i, int j, T a) {
        const T h = A::neg(A::add(Y[(int64_t)i * n + j], a));
        fac[nd_at(sf, N.row_f + s + j, i)] = h;
        fac[nd_at(sb, N.row_b + i, j)] = h;
    });
    __syncthreads();
    for (int t = tid; t < b * b; t += nt) {
        const int i = t / b, j = t - i * b;
        T* d = F + (int64_t)(s + i) * n + s + j;
        T a = *d;
        const T* h = fac + nd_at(sf, N.row_f + s + j, 0);
        for (int k = 0; k < s; ++k) a = A::fma_(F[(int64_t)(s + i) * n + k], h[(k >> 2) * 128 + (k & 3)], a);
        *d = a;
    }
}

NdTables nd_tables(const thm_mesh* m) {
    const auto& D = m->ndd;
    NdTables T{};
    T.parts = D.parts.p; T.levs = D.levs.p; T.slt = D.slt.p;
    T.rowd = D.rowd.p; T.rowm = D.rowm.p; T.ymap = D.ymap.p; T.rmap = D.rmap.p;
    T.idx = D.idx.p; T.perm = D.perm.p; T.welem = D.welem.p; T.subs = m->d_subs.p;
    T.mw = m->nd.mw;
    return T;
}

void require_nd(const thm_mesh* m) {
    THM_REQUIRE(m->nd_ok, "subdomain too large for the shared-memory block solve");
}

template <class T>
static void factor(thm_sys* s, DArr<T>& fac, const char* what) {
    const thm_mesh* m = s->m;
    const NdHost& H = m->nd;
    cudaStream_t st = s->st;
    require_nd(m);
    fac.alloc(H.fac_elems);
    fac.zero(st);
    int64_t most[2] = {0, 0};
    const int nd = (int)H.depth_front.size();
    for (int d = 0; d < nd; ++d) most[d & 1] = std::max(most[d & 1], H.depth_front[d]);
    DArr<T> front[2], aux;
    front[0].alloc(most[0]);
    front[1].alloc(most[1]);
    aux.alloc(3 * std::max(most[0], most[1]));
    DArr<int> status;
    status.alloc(1);
    status.zero(st);
    const size_t cap = 200 * 1024;
    THM_CUDA(cudaFuncSetAttribute(k_nd_factor<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
    for (int d = 0; d < nd; ++d) {
        const int64_t n0 = H.depth_node[d], cnt = H.depth_node[d + 1] - n0;
        const int ms = std::max(1, H.depth_s[d]), mn = H.depth_n[d];
        // blocks up to smem_s in shared memory; the others of the depth in place
        const int smem_s = (size_t)ms * ms * sizeof(T) <= cap ? ms : 0;
        const size_t smem = (size_t)2 * ms * sizeof(T) + (size_t)smem_s * smem_s * sizeof(T) + (size_t)ms * sizeof(int);
        int threads = 32;
        while (threads < 512 && threads * 16 < mn * mn) threads *= 2;
        THM_LAUNCH(THM_K_SETUP, st, k_nd_factor<T><<<(unsigned)cnt, threads, smem, st>>>(
            nd_tables(m), m->ndd.nodes.p, n0, m->ndd.rows.p, m->ndd.cmap.p, m->ndd.childs.p, H.C, smem_s, ms,
            m->d_slice_ptr.p, m->d_sell_col.p, m->d_sell_pad.p, s->val64.p, s->bg64.p, s->bs64.p, front[d & 1].p,
            front[(d + 1) & 1].p, aux.p, fac.p, status.p));
        THM_CUDA(cudaGetLastError());
    }
    std::vector<int> hs;
    status.download(hs, st);
    if (hs[0] != 0) fail(THM_ESINGULAR, what);
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
