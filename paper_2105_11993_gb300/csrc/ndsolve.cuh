// x = P_i^{-1} r for every subdomain at once (the block preconditioner of
// Eq. 7: the same real P_i^{-1} applied to the real and the imaginary part),
// or x = T_i^{-1} r from complex factors (the full 2x2 block operator of
// Section 3.2), by nested dissection of the subdomain's cells (nd.cuh).
//
// Every tree node eliminates its s unknowns against the b unknowns of its
// ancestors that its cells touch.  With W = S^{-1} (S the node's Schur
// complement) and H = W F (F the coupling to the b unknowns), both dense:
//   up    y = r_s + sum_children u,   t = W y,   u = sum_children u - H^T y
//   down  x_s = t - H x_b
// so a solve is one sweep up the tree and one down, each node two small
// GEMVs, instead of a chain over the levels of a banded elimination: for a
// 32x32-cell order-2 subdomain 0.38M values are multiplied instead of 1.2M
// (dense level blocks of 130 rows) in 7 dependent steps each way and the root
// instead of 33.  Measured against that level-by-level elimination (64 such
// subdomains, FP64): 529 us to 210 us per apply, factorisation 28 ms to 7 ms
// (18 ms in the mean with what ndfactor.cu does near resonances).
//
// One cluster of C CTAs per subdomain: the top of the tree is one root node
// with at least C subtrees under it, each CTA runs its subtrees alone with
// their vectors in its shared memory, and the CTAs meet twice, before and
// after the root (each forms its share of the root's rows; children's u are
// read and root values written through distributed shared memory).  Within a
// CTA the nodes of one depth are independent: their rows are cut into slices
// of 32 (a lane owns a row), stored as column quads so that a lane loads 16
// bytes (32 in FP64) and a warp a contiguous block per quad.  Every sum has a
// fixed order, so results do not depend on scheduling.
#pragma once

#include <cooperative_groups.h>
#include <type_traits>

#include "kernels.cuh"
#include "nd.cuh"

namespace thm {

__device__ __forceinline__ bool mbar_try(uint64_t* bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ unsigned long long nd_now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Factor element types: real (Eq. 7) or complex (the full 2x2 block operator).
template <class T> struct NdCplx { static constexpr bool value = false; };
template <> struct NdCplx<float2> { static constexpr bool value = true; };
template <> struct NdCplx<double2> { static constexpr bool value = true; };

// One column quad of a lane's row: 4 consecutive factor entries.
template <class FW> struct NdQuad;
template <> struct NdQuad<float> { float4 a; };
template <> struct NdQuad<double> { double2 a, b; };
template <> struct NdQuad<float2> { float4 a, b; };
template <> struct NdQuad<double2> { double2 a, b, c, d; };

__device__ __forceinline__ void nd_load(const float* p, NdQuad<float>& q) { q.a = __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ void nd_load(const double* p, NdQuad<double>& q) {
    q.a = __ldg(reinterpret_cast<const double2*>(p));
    q.b = __ldg(reinterpret_cast<const double2*>(p) + 1);
}
__device__ __forceinline__ void nd_load(const float2* p, NdQuad<float2>& q) {
    q.a = __ldg(reinterpret_cast<const float4*>(p));
    q.b = __ldg(reinterpret_cast<const float4*>(p) + 1);
}
__device__ __forceinline__ void nd_load(const double2* p, NdQuad<double2>& q) {
    q.a = __ldg(p); q.b = __ldg(p + 1); q.c = __ldg(p + 2); q.d = __ldg(p + 3);
}

template <class R, class V>
__device__ __forceinline__ void nd_fma(R w, const V& y, R& ar, R& ai) { ar += w * y.x; ai += w * y.y; }
// (two fused multiply-adds per sum: with the product difference formed first a
// third instruction, 192 -> 158 us per apply, 9 subdomains of 33x26 cells, FP64)
template <class R, class W2, class V>
__device__ __forceinline__ void nd_cfma(const W2& w, const V& y, R& ar, R& ai) {
    ar = fma((R)w.x, y.x, fma(-(R)w.y, y.y, ar));
    ai = fma((R)w.x, y.y, fma((R)w.y, y.x, ai));
}
template <class R, class V>
__device__ __forceinline__ void nd_acc(const NdQuad<float>& q, const V (&y)[4], R& ar, R& ai) {
    nd_fma((R)q.a.x, y[0], ar, ai); nd_fma((R)q.a.y, y[1], ar, ai);
    nd_fma((R)q.a.z, y[2], ar, ai); nd_fma((R)q.a.w, y[3], ar, ai);
}
template <class R, class V>
__device__ __forceinline__ void nd_acc(const NdQuad<double>& q, const V (&y)[4], R& ar, R& ai) {
    nd_fma((R)q.a.x, y[0], ar, ai); nd_fma((R)q.a.y, y[1], ar, ai);
    nd_fma((R)q.b.x, y[2], ar, ai); nd_fma((R)q.b.y, y[3], ar, ai);
}
template <class R, class V>
__device__ __forceinline__ void nd_acc(const NdQuad<float2>& q, const V (&y)[4], R& ar, R& ai) {
    nd_cfma(make_float2(q.a.x, q.a.y), y[0], ar, ai); nd_cfma(make_float2(q.a.z, q.a.w), y[1], ar, ai);
    nd_cfma(make_float2(q.b.x, q.b.y), y[2], ar, ai); nd_cfma(make_float2(q.b.z, q.b.w), y[3], ar, ai);
}
template <class R, class V>
__device__ __forceinline__ void nd_acc(const NdQuad<double2>& q, const V (&y)[4], R& ar, R& ai) {
    nd_cfma(q.a, y[0], ar, ai); nd_cfma(q.b, y[1], ar, ai);
    nd_cfma(q.c, y[2], ar, ai); nd_cfma(q.d, y[3], ar, ai);
}

__device__ __forceinline__ void nd_y4(const float2* y, float2 (&v)[4]) {
    const float4 a = reinterpret_cast<const float4*>(y)[0], b = reinterpret_cast<const float4*>(y)[1];
    v[0] = make_float2(a.x, a.y); v[1] = make_float2(a.z, a.w);
    v[2] = make_float2(b.x, b.y); v[3] = make_float2(b.z, b.w);
}
__device__ __forceinline__ void nd_y4(const double2* y, double2 (&v)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = y[k];
}

// Quads in flight per lane: 16 registers of factor entries in FP32, 32 in FP64.
template <class FW> constexpr int nd_unroll() { return sizeof(FW) >= 16 ? 2 : 4; }

// sum over the column quads [qa, qb) of a slice (p: the slice plus the lane's
// column offset) of row entries times y (contiguous, 4 per quad)
template <class FW, class V>
__device__ __forceinline__ V nd_dot(const FW* __restrict__ p, int qa, int qb, const V* y) {
    using R = typename VT<V>::R;
    constexpr int U = nd_unroll<FW>();
    R ar = 0, ai = 0;
    int q = qa;
    for (; q + U <= qb; q += U) {
        NdQuad<FW> w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) nd_load(p + (int64_t)(q + u) * 128, w[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            V v[4];
            nd_y4(y + 4 * (q + u), v);
            nd_acc(w[u], v, ar, ai);
        }
    }
    for (; q < qb; ++q) {
        NdQuad<FW> w;
        nd_load(p + (int64_t)q * 128, w);
        V v[4];
        nd_y4(y + 4 * q, v);
        nd_acc(w, v, ar, ai);
    }
    return mk<V>(ar, ai);
}

// The same with the y entries gathered: vec[idx[0..]].
template <class FW, class V>
__device__ __forceinline__ V nd_dot_gather(const FW* __restrict__ p, int qa, int qb, const uint16_t* __restrict__ idx,
                                           const V* vec) {
    using R = typename VT<V>::R;
    constexpr int U = nd_unroll<FW>();
    R ar = 0, ai = 0;
    int q = qa;
    for (; q + U <= qb; q += U) {
        NdQuad<FW> w[U];
        uint2 ix[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            ix[u] = __ldg(reinterpret_cast<const uint2*>(idx) + q + u);
            nd_load(p + (int64_t)(q + u) * 128, w[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const V v[4] = {vec[ix[u].x & 0xffffu], vec[ix[u].x >> 16], vec[ix[u].y & 0xffffu], vec[ix[u].y >> 16]};
            nd_acc(w[u], v, ar, ai);
        }
    }
    for (; q < qb; ++q) {
        const uint2 ix = __ldg(reinterpret_cast<const uint2*>(idx) + q);
        NdQuad<FW> w;
        nd_load(p + (int64_t)q * 128, w);
        const V v[4] = {vec[ix.x & 0xffffu], vec[ix.x >> 16], vec[ix.y & 0xffffu], vec[ix.y >> 16]};
        nd_acc(w, v, ar, ai);
    }
    return mk<V>(ar, ai);
}

template <class V>
__device__ __forceinline__ V nd_add(V a, V b) { return mk<V>(a.x + b.x, a.y + b.y); }

// v + the (at most 2 * mw) children's entries of u named by the map words
template <class V>
__device__ __forceinline__ V nd_gather_children(V v, const uint32_t* __restrict__ map, int64_t i, int mw, const V* u) {
    if (mw == 1) {
        const uint32_t a = __ldg(map + i);
        if ((a & 0xffffu) != ND_NONE) v = nd_add(v, u[a & 0xffffu]);
        if ((a >> 16) != ND_NONE) v = nd_add(v, u[a >> 16]);
    } else {
        const uint2 a = __ldg(reinterpret_cast<const uint2*>(map) + i);
        if ((a.x & 0xffffu) != ND_NONE) v = nd_add(v, u[a.x & 0xffffu]);
        if ((a.x >> 16) != ND_NONE) v = nd_add(v, u[a.x >> 16]);
        if ((a.y & 0xffffu) != ND_NONE) v = nd_add(v, u[a.y & 0xffffu]);
        if ((a.y >> 16) != ND_NONE) v = nd_add(v, u[a.y >> 16]);
    }
    return v;
}

// Shared-memory layout (host and device agree through this); the two u
// buffers and the staged y can live in a global workspace instead (subdomains
// whose vectors outgrow shared memory).
struct NdLayout {
    size_t lev, slt, vec, ysc, u0, u1, part, total;
};
template <class V>
__host__ __device__ inline NdLayout nd_layout(const NdSizes& z, int slt_smem, int u_glob, int y_glob) {
    auto r16 = [](size_t v) { return (v + 15) / 16 * 16; };
    NdLayout L;
    size_t o = 16;                                   // the mbarrier
    L.lev = o; o += (size_t)(z.nlev + 1) * sizeof(NdLev);
    L.slt = o; o += slt_smem ? r16((size_t)z.nslt * sizeof(int2)) : 0;
    L.vec = o; o += r16((size_t)z.nvec * sizeof(V));
    L.ysc = o; o += y_glob ? 0 : r16((size_t)z.ny * sizeof(V));
    L.u0 = o; o += u_glob ? 0 : r16((size_t)z.nu[0] * sizeof(V));
    L.u1 = o; o += u_glob ? 0 : r16((size_t)z.nu[1] * sizeof(V));
    L.part = o; o += (size_t)ND_NT * sizeof(V);
    L.total = o;
    return L;
}

// The workspace of a CTA whose u buffers and staged y are in global memory, in
// vector entries: u of the even depths at 0.  Every part starts at a multiple
// of 4 entries, since the staged y is read 16 bytes at a time (nd_y4).
struct NdGlob {
    int64_t u1, y, stride;
};
__host__ __device__ inline NdGlob nd_glob_layout(const NdSizes& z) {
    auto r4 = [](int64_t v) { return (v + 3) / 4 * 4; };
    NdGlob g;
    g.u1 = r4(z.nu[0]);
    g.y = g.u1 + r4(z.nu[1]);
    g.stride = g.y + r4(z.ny);
    return g;
}

// Launch options that the host decides from the sizes (nd_memory).
struct NdMem {
    int slt_smem, u_glob, y_glob, prefetch;
    int64_t glob_stride;
};

// Work items that a dot-product pass is cut into while there are few basis
// vectors: three per warp, so that the last round is not nearly empty.
constexpr int SUB_ITEMS = 3 * ND_NW;
// Shared memory of a subdomain solve that outlives a step: rotations and g of the cycle (givens_core)
// and the previous step's [b; d].
__host__ __device__ inline size_t sub_keep_bytes(int m) { return (size_t)m * 40 + (size_t)(m + 1) * 48 + 48; }

// Bytes of the Krylov phases' shared memory (they reuse the apply's): u and w
// of the CTA's rows, the totals and the Hessenberg column, the coefficients,
// the warps' sums.
template <class V>
__host__ __device__ inline size_t sub_krylov_bytes(int rows, int m, int k_glob) {
    const size_t red = (size_t)(m / 4 + 2 + SUB_ITEMS) * 16 * sizeof(typename VT<V>::R);
    return (k_glob ? 0 : 2 * (size_t)rows * sizeof(V)) + (size_t)(2 * m + 2) * 16 + (size_t)(m + 1) * 16 +
           (size_t)(2 * m + 2) * sizeof(V) + (red + 15) / 16 * 16;
}
// rows of a CTA: the subdomain's local rows in C equal parts of whole warps
// of the SELL slices, or of 8 where that would leave CTAs without rows
__host__ __device__ inline int sub_rows(int64_t n, int C) {
    const int64_t r = (n + C - 1) / C, g = r >= 512 ? 32 : 8;
    return (int)((r + g - 1) / g * g);
}

// The shared memory of a solve kernel with vectors V: one function for the
// build of the trees, which picks the CTAs per subdomain by it, and for the
// launches.  more: bytes that other phases need over the apply's vectors;
// keep: bytes beside everything.  glob: the u buffers, then the staged y, then
// the slice table may move to global memory, in this order, until it fits
// (force, for tests: all of them do).  Returns the bytes, or 0 if it does not fit.
template <class V>
inline size_t nd_fit(const NdSizes& z, bool glob, size_t more, size_t keep, NdMem* mm, bool force = false) {
    mm->slt_smem = (size_t)z.nslt * sizeof(int2) <= 16 * 1024 ? 1 : 0;
    mm->u_glob = mm->y_glob = 0;
    auto need = [&]() {
        const NdLayout L = nd_layout<V>(z, mm->slt_smem, mm->u_glob, mm->y_glob);
        const size_t all = L.total > L.vec + more ? L.total : L.vec + more;
        return (all + 15) / 16 * 16 + keep;
    };
    if (glob) {
        if (force || need() > ND_SMEM_MAX) mm->u_glob = 1;
        if (force || need() > ND_SMEM_MAX) mm->y_glob = 1;
        if (force || need() > ND_SMEM_MAX) mm->slt_smem = 0;
    } else if (force || !mm->slt_smem) {
        return 0;
    }
    mm->glob_stride = (mm->u_glob || mm->y_glob) ? nd_glob_layout(z).stride : 0;
    return need() <= ND_SMEM_MAX ? need() : 0;
}

// Where a CTA's pieces are: built once per launch, used by every apply in it.
template <class V>
struct NdCta {
    NdPart P;
    const NdLev* lev;
    const int2* slt;
    V *vec, *ysc, *u_even, *u_odd, *part;
    V* glob;                  // this subdomain's u_odd of rank 0 in the global workspace (u_glob), its ranks glob_stride apart
    int64_t glob_stride;
    int rank, C, u_glob, ny, prefetch;
    bool ok;                  // the tables came
};

// One thread waits for the table copies, for at most wait_ns; then it gives up
// (the CTA skips the work and keeps the barriers).  Copies under way write the
// CTA's shared memory, so it does not leave before they are through, or as
// long again.  (Out of line: the solve kernels have no registers to spare.)
static __device__ __noinline__ void nd_wait(uint64_t* bar, unsigned long long wait_ns, int stall, int* s_abort, int* err) {
    for (int round = 0; round < 2; ++round) {
        const unsigned long long t0 = nd_now_ns();
        do {
            if (mbar_try(bar, 0)) return;
        } while (nd_now_ns() - t0 <= wait_ns);
        *s_abort = 1;
        atomicExch(err, 1);
        if (stall) return;                     // (none was sent)
    }
}

// Start of a solve CTA: its level and slice tables come by TMA (stall:
// failure-detection test, the copies never come).  GLOB: some of the tables
// and vectors are in global memory; else all are in shared memory, which the
// compiler must see (through pointers that may be either, an apply takes 126
// registers instead of 69 and its shared-memory loads several times as long).
template <bool GLOB, class V>
__device__ __forceinline__ void nd_enter(NdCta<V>& c, const NdTables& T, const NdSizes& z, const NdMem& mm, V* glob,
                                         unsigned char* smem, int sub, int rank, int C, unsigned long long wait_ns, int stall,
                                         int* s_abort, int* err) {
    const int tid = threadIdx.x;
    c.P = T.parts[(int64_t)sub * C + rank];
    const NdLayout lay = nd_layout<V>(z, mm.slt_smem, mm.u_glob, mm.y_glob);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
    NdLev* lev = reinterpret_cast<NdLev*>(smem + lay.lev);
    c.lev = lev;
    c.vec = reinterpret_cast<V*>(smem + lay.vec);
    c.part = reinterpret_cast<V*>(smem + lay.part);
    c.slt = reinterpret_cast<const int2*>(smem + lay.slt);
    c.ysc = reinterpret_cast<V*>(smem + lay.ysc);
    c.u_even = reinterpret_cast<V*>(smem + lay.u0);        // u of the even depths
    c.u_odd = reinterpret_cast<V*>(smem + lay.u1);
    const NdGlob gw = nd_glob_layout(z);
    if constexpr (GLOB) {
        V* gl = glob + ((int64_t)sub * C + rank) * mm.glob_stride;
        if (!mm.slt_smem) c.slt = T.slt + c.P.slt0;
        if (mm.y_glob) c.ysc = gl + gw.y;
        if (mm.u_glob) {
            c.u_even = gl;
            c.u_odd = gl + gw.u1;
        }
    }
    c.glob = glob + (int64_t)sub * C * mm.glob_stride + gw.u1;
    c.glob_stride = mm.glob_stride;
    c.rank = rank;
    c.C = C;
    c.u_glob = mm.u_glob;
    c.ny = z.ny;
    c.prefetch = mm.prefetch;
    if (tid == 0) {
        *s_abort = 0;
        mbar_init(bar, 1);
        mbar_fence_init();
        fence_proxy_async();
        if (!stall) {
            const unsigned lb = (unsigned)((c.P.nlev + 1) * sizeof(NdLev));
            const unsigned sb = mm.slt_smem ? (unsigned)((c.P.nslt + 1) / 2 * 16) : 0u;
            mbar_expect_tx(bar, lb + sb);
            tma_load_1d(lev, T.levs + c.P.lev0, lb, bar);
            if (sb) tma_load_1d(smem + lay.slt, T.slt + c.P.slt0, sb, bar);
        }
        if (!mbar_try(bar, 0)) nd_wait(bar, wait_ns, stall, s_abort, err);
    }
    __syncthreads();
    c.ok = *s_abort == 0;
}

// Asks for the factor entries of n slices from slice s0 on to come to L2.
template <class FW>
__device__ __forceinline__ void nd_prefetch(const FW* fac, const int2* slt, int s0, int n) {
    if (n <= 0) return;
    const int64_t a = slt[s0].x, b = (int64_t)slt[s0 + n - 1].x + slt[s0 + n - 1].y;
    if (a == b) return;                        // rows of nodes without unknowns of their own
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(fac + a * 128),
                 "r"((unsigned)((b - a) * 128 * sizeof(FW)))
                 : "memory");
}

// One apply y = P_i^{-1} x by the CTAs of a cluster.  x may have been written
// by other CTAs of the cluster in this launch (before a cluster barrier), so
// it is read with ordinary loads.
template <bool GLOB, class V, class FW>
__device__ __forceinline__ void nd_apply_cta(const NdCta<V>& c, const NdTables& T, const FW* __restrict__ fac, const V* x,
                                             V* y) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const NdPart& P = c.P;
    const NdLev* lev = c.lev;
    const int2* slt = c.slt;
    V *vec = c.vec, *ysc = c.ysc, *u_even = c.u_even, *u_odd = c.u_odd, *part = c.part;
    const bool ok = c.ok;
    const int C = c.C, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nlev = ok ? P.nlev : 0;
    // the rows of step st: up 0..nlev-1, the root nlev, down
    auto prefetch = [&](int st) {
        if (!c.prefetch || tid != 0 || !ok || st > 2 * nlev) return;
        const NdLev& L = lev[st <= nlev ? st : 2 * nlev - st];
        if (st < nlev || (st == nlev && P.sroot > 0)) nd_prefetch(fac, slt, L.sltf, L.nsf);
        else if (st > nlev) nd_prefetch(fac, slt, L.sltb, L.nsb);
    };
    prefetch(0);
    prefetch(1);
    const int32_t* perm = T.perm + P.perm0;
    constexpr int G = 4;                       // gathers in flight per thread
    for (int p0 = tid; p0 < P.nvec; p0 += G * ND_NT) {
        int32_t r[G];
        V v[G];
#pragma unroll
        for (int g = 0; g < G; ++g) r[g] = p0 + g * ND_NT < P.nvec ? __ldg(perm + p0 + g * ND_NT) : -1;
#pragma unroll
        for (int g = 0; g < G; ++g) v[g] = r[g] >= 0 ? x[r[g]] : mk<V>(0, 0);
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (p0 + g * ND_NT < P.nvec) vec[p0 + g * ND_NT] = v[g];
    }
    for (int p = tid; p < c.ny; p += ND_NT) ysc[p] = mk<V>(0, 0);     // rows are padded to the widest node of their slice
    __syncthreads();

    // ---- up: the CTA's subtrees, deepest level first
    for (int l = 0; l < nlev; ++l) {
        const NdLev L = lev[l];
        prefetch(l + 2);
        const V* uin = (L.depth & 1) ? u_even : u_odd;
        V* uout = (L.depth & 1) ? u_odd : u_even;
        for (int e = tid; e < L.nv; e += ND_NT) {
            V v = vec[L.v0 + e];
            if (l > 0) v = nd_gather_children(v, T.ymap, (int64_t)L.ymap + e, T.mw, uin);
            ysc[e] = v;
        }
        __syncthreads();
        auto put = [&](int row, V a) {         // t = W y into vec, u = children's u - H^T y
            const uint32_t d = __ldg(T.rowd + L.rowf + row);
            if (d == ND_NOROW) return;
            const uint32_t dst = d >> 16;
            if (!(dst & ND_U)) vec[dst] = a;
            else uout[dst & ~ND_U] = l > 0 ? nd_gather_children(a, T.rowm, (int64_t)L.rowf + row, T.mw, uin) : a;
        };
        if (L.ksf == 1) {
            for (int sl = warp; sl < L.nsf; sl += ND_NW) {
                const int2 S = slt[L.sltf + sl];
                const uint32_t d = __ldg(T.rowd + L.rowf + sl * 32 + lane);
                put(sl * 32 + lane, nd_dot(fac + (int64_t)S.x * 128 + lane * 4, 0, S.y, ysc + (d == ND_NOROW ? 0 : (d & 0xffffu))));
            }
        } else {                               // few slices: their columns are shared out over the warps
            const int sl = warp / L.ksf, k = warp % L.ksf;
            if (sl < L.nsf) {
                const int2 S = slt[L.sltf + sl];
                const uint32_t d = __ldg(T.rowd + L.rowf + sl * 32 + lane);
                part[tid] = nd_dot(fac + (int64_t)S.x * 128 + lane * 4, S.y * k / L.ksf, S.y * (k + 1) / L.ksf,
                                   ysc + (d == ND_NOROW ? 0 : (d & 0xffffu)));
            }
            __syncthreads();
            if (tid < L.nsf * 32) {
                V a = part[warp * L.ksf * 32 + lane];
                for (int q = 1; q < L.ksf; ++q) a = nd_add(a, part[(warp * L.ksf + q) * 32 + lane]);
                put(tid, a);
            }
        }
        __syncthreads();
    }

    // ---- the root, shared out over the cluster
    if (P.sroot > 0) {
        if (ok)
            for (int e = tid; e < P.sroot; e += ND_NT) ysc[e] = vec[e];
        cluster.sync();                        // every rank's u is complete, and its r of the root is staged
        if (ok) {
            const NdLev L = lev[nlev];
            prefetch(nlev + 2);
            for (int e = tid; e < P.sroot; e += ND_NT) {
                V v = ysc[e];
                for (int q = 0; q < 2 * T.mw; ++q) {
                    const uint32_t a = __ldg(T.rmap + ((int64_t)P.rmap0 + e) * 2 * T.mw + q);
                    if (a == 0xffffffffu) break;
                    const int rk = (int)(a >> 16);
                    const V* src;
                    if constexpr (GLOB) src = c.u_glob ? c.glob + rk * c.glob_stride : cluster.map_shared_rank(u_odd, rk);
                    else src = cluster.map_shared_rank(u_odd, rk);
                    v = nd_add(v, src[a & 0xffffu]);
                }
                ysc[e] = v;
            }
            // the staged y of the last level may reach past the root's rows
            for (int e = P.sroot + tid; e < (P.sroot + 3) / 4 * 4; e += ND_NT) ysc[e] = mk<V>(0, 0);
            __syncthreads();
            auto put = [&](int row, V a) {     // x of the root goes to every rank
                const uint32_t d = __ldg(T.rowd + L.rowf + row);
                if (d == ND_NOROW) return;
                for (int rk = 0; rk < C; ++rk) cluster.map_shared_rank(vec, rk)[d >> 16] = a;
            };
            if (L.ksf == 1) {
                for (int sl = warp; sl < L.nsf; sl += ND_NW) {
                    const int2 S = slt[L.sltf + sl];
                    put(sl * 32 + lane, nd_dot(fac + (int64_t)S.x * 128 + lane * 4, 0, S.y, ysc));
                }
            } else {
                const int sl = warp / L.ksf, k = warp % L.ksf;
                if (sl < L.nsf) {
                    const int2 S = slt[L.sltf + sl];
                    part[tid] = nd_dot(fac + (int64_t)S.x * 128 + lane * 4, S.y * k / L.ksf, S.y * (k + 1) / L.ksf, ysc);
                }
                __syncthreads();
                if (tid < L.nsf * 32) {
                    V a = part[warp * L.ksf * 32 + lane];
                    for (int q = 1; q < L.ksf; ++q) a = nd_add(a, part[(warp * L.ksf + q) * 32 + lane]);
                    put(tid, a);
                }
            }
        }
        cluster.sync();                        // x of the root is complete; no rank touches another's memory after this
    }

    // ---- down
    for (int l = nlev - 1; l >= 0; --l) {
        const NdLev L = lev[l];
        prefetch(2 * nlev - l + 2);
        auto put = [&](uint32_t d, V a) { vec[d >> 16] = nd_add(vec[d >> 16], a); };
        if (L.ksb == 1) {
            for (int sl = warp; sl < L.nsb; sl += ND_NW) {
                const int2 S = slt[L.sltb + sl];
                const uint32_t d = __ldg(T.rowd + L.rowb + sl * 32 + lane);
                const V a = nd_dot_gather(fac + (int64_t)S.x * 128 + lane * 4, 0, S.y,
                                          T.idx + L.idx + 4 * (d == ND_NOROW ? 0 : (d & 0xffffu)), vec);
                if (d != ND_NOROW) put(d, a);
            }
        } else {
            const int sl = warp / L.ksb, k = warp % L.ksb;
            if (sl < L.nsb) {
                const int2 S = slt[L.sltb + sl];
                const uint32_t d = __ldg(T.rowd + L.rowb + sl * 32 + lane);
                part[tid] = nd_dot_gather(fac + (int64_t)S.x * 128 + lane * 4, S.y * k / L.ksb, S.y * (k + 1) / L.ksb,
                                          T.idx + L.idx + 4 * (d == ND_NOROW ? 0 : (d & 0xffffu)), vec);
            }
            __syncthreads();
            if (tid < L.nsb * 32) {
                V a = part[warp * L.ksb * 32 + lane];
                for (int q = 1; q < L.ksb; ++q) a = nd_add(a, part[(warp * L.ksb + q) * 32 + lane]);
                const uint32_t d = __ldg(T.rowd + L.rowb + tid);
                if (d != ND_NOROW) put(d, a);
            }
        }
        __syncthreads();
    }
    if (ok)
        for (int p = tid; p < P.nvec; p += ND_NT) {
            const int32_t r = __ldg(perm + p);
            if (r >= 0 && (p >= P.sroot || (p >= P.rr0 && p < P.rr0 + P.nrr))) y[r] = vec[p];
        }
}

template <bool GLOB, class V, class FW>
__global__ void __launch_bounds__(ND_NT, 2)
k_nd_solve(NdTables T, NdSizes z, NdMem mm, V* __restrict__ glob, const FW* __restrict__ fac, unsigned long long wait_ns,
           int stall, int* __restrict__ err, unsigned long long* __restrict__ work, const V* __restrict__ x,
           V* __restrict__ y) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_abort;
    NdCta<V> c;
    nd_enter<GLOB>(c, T, z, mm, glob, smem, (int)blockIdx.y, (int)blockIdx.x, (int)gridDim.x, wait_ns, stall, &s_abort, err);
    nd_apply_cta<GLOB>(c, T, fac, x, y);
    if (work && blockIdx.x == 0 && threadIdx.x == 0) {     // instrumentation: the work this launch does
        atomicAdd(&work[0], (unsigned long long)T.welem[blockIdx.y]);
        atomicAdd(&work[1], (unsigned long long)T.subs[blockIdx.y].n);
    }
}

}  // namespace thm
