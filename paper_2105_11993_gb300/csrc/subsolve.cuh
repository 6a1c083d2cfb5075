// The subdomain solves T_i x_i = b_i of a sweep, each from start to end in one
// cluster of one launch: block-preconditioned flexible GMRES with delayed
// re-orthogonalisation (DCGS2), restarted on the FP64 residual.
//
// A subdomain's solve depends on no other, so its cluster runs every Arnoldi
// step itself: preconditioner apply (ndsolve.cuh), operator apply, one pass of
// dot products and one update pass over the basis, the scalar step and the
// stopping test, with cluster barriers between them.  Step by step as kernels
// over all subdomains (5 launches and a monitor copy per step) a step of the
// 32x32 order-1 problem took 230 us, nearly all of it launch and tail latency;
// in this kernel a step takes about 45 us.  Whole solves, before and after
// (with the shorter scalar step of krylov.cuh and the interface passes there):
// 32x32 order 1 FP64 1315 -> 219 ms, 48x48 order 2 mixed 978 -> 611 ms, the
// gradient of a 6^3 cube 1900 -> 809 ms; one sweep of 64 subdomains of 8^3
// cells 25.3 -> 15.9 ms, of 64 of 32^2 cells order 2 mixed 26.4 -> 25.2 ms, of
// 16 of 32^2 cells order 2 FP64 49 -> 39 ms (58 ms while the sums of products
// were written a * b + c * d added to the sum, which compiles to a multiply, a
// fused multiply-add and an addition: three FP64 instructions instead of two).
// What bounds it: latencies (a cluster barrier about 1k cycles, an L2 load
// 700 to 1200, the scalar step's FP64 chain 5 to 10k) on small subdomains;
// on large ones the factor stream and, in FP64, the FP64 units (2 FMA per
// clock and SM): the Gram-Schmidt passes of step 36 alone are
// 300k cycles of multiply-adds.
//
// FP64 (V = double2): cycles of at most m steps until the residual is below
// tol ||b|| (or fails to halve over a cycle).  Mixed (V = float2): each cycle
// solves T d = r in FP32 to cycle_tol of its own right-hand side and x and r
// are kept in FP64.
//
// Step j of a cycle holds the orthonormal v_0..v_{j-1} and, in basis slot j,
// u_j: the next vector orthogonalised once.  z_j = M u_j (kept), w_j = A z_j.
// One pass over the basis gives s = V^H u_j, b = V^H w_j, c1 = u_j^H u_j and
// c2 = u_j^H w_j, and then
//     gamma_j = sqrt(c1 - |s|^2),      v_j = (u_j - V s) / gamma_j,
//     d_j     = v_j^H w_j = (c2 - s^H b) / gamma_j,
//     u_{j+1} = (w_j - V b - v_j d_j) / gamma_j
//             = w_j / gamma_j - u_j d_j / gamma_j^2 - V (b - s d_j / gamma_j) / gamma_j,
// which the second pass writes (v_j over u_j in slot j, u_{j+1} into slot
// j + 1).  (Without the division by gamma_j the norms of the u_j grow
// geometrically, ~1e13 after 40 steps, and the cycle loses its accuracy;
// with it |u_{j+1}| is about h_{j+1,j}.)  One step later
// u_{j+1} = V_{0..j} s_{j+1} + gamma_{j+1} v_{j+1}, so
//     A z_j = V_{0..j} ([b_j; d_j] + gamma_j s_{j+1}) + gamma_j gamma_{j+1} v_{j+1}:
// Hessenberg column j becomes final at step j + 1, where its Givens step and
// the residual test run.  The directions z_j span the same space as the
// M v_j, and x = x_0 + Z y minimises the residual over it as in flexible
// GMRES.  v_0 = r / ||r|| is taken as it is (gamma_0 = 1); a cycle of m
// columns ends with a step that only finalises column m - 1 (no M, no A).
#pragma once

#include "krylov.cuh"
#include "ndsolve.cuh"

namespace thm {

// Device totals of the solves since they were last zeroed.
struct SolveTotals {
    unsigned long long iters, dof_iters;   // Arnoldi steps, times the subdomain's DOFs
    int max_iters;                         // largest count of one FP64 solve, or of one FP32 cycle
    int no_conv, breakdown;                // FP64 solves that hit maxit; non-finite projections (FP64)
    int pad;
};

template <class V, class F>
struct SubArgs {
    int m, maxit, max_cycles;
    double tol, cycle_tol;
    int col16;
    int64_t n;                  // local DOFs of all subdomains: stride of the basis vectors
    const double2* b;
    double2 *x, *r;             // solution; residual (workspace)
    V *basis, *zbasis, *w;
    double2* partial;           // [n_sub * C][2m + 2]
    double2* y;                 // [n_sub][m]
    GivensArgs g;
    const Sub* subs;
    const int64_t* slice_ptr;
    const int32_t* col;
    const uint16_t* col_rel;
    SpmvMat<F> A;
    SpmvMat<double> A64;
    SolveTotals* totals;
    unsigned long long *kw, *kw64, *bt;     // work counters: SpMV rows, dot and update bytes; FP64 SpMV rows; applies
};

// A sum with the rounding of its partial sums compensated (Kahan): FP32 sums
// over a CTA's rows stay as accurate as sums over 8 rows.  FP64 sums plainly.
template <class R> struct RowSum;
template <> struct RowSum<float> {
    float s = 0, c = 0;
    __device__ __forceinline__ void add(float v) {
        const float y = __fsub_rn(v, c), t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
};
template <> struct RowSum<double> {
    double s = 0;
    __device__ __forceinline__ void add(double v) { s += v; }
};

// Row r of a product with the subdomain operator, x: the vector over all subdomains
template <bool GLOB, class VX, class FA, class V, class F>
__device__ __forceinline__ VX sub_spmv(const SubArgs<V, F>& a, const SpmvMat<FA>& A, int64_t r, const VX* x, int64_t off) {
    // (subdomains of more than 65,536 DOFs have no 16-bit columns: their solves run as GLOB)
    if (!GLOB || a.col16) return spmv_row<VX, FA, uint16_t>(r, a.slice_ptr, a.col_rel, A, 1, x + off, off);
    return spmv_row<VX, FA, int32_t>(r, a.slice_ptr, a.col, A, 1, x, 0);
}

// Sums of K values per thread over the cluster, the same in every CTA (fixed
// order).  Two buffers in turn: a CTA writes a buffer again only after the
// barrier of the other's sum, which every CTA reaches after its reads.
template <int K>
__device__ __forceinline__ void cluster_sum(double (&v)[K], int& turn, int rank, int C) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ double s_warp[ND_NW][K];
    __shared__ double s_cl[2][8][K];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) s_warp[warp][k] = v[k];
    __syncthreads();
    if ((int)threadIdx.x < C) {
        double* dst = cluster.map_shared_rank(&s_cl[turn][rank][0], (int)threadIdx.x);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            double t = 0;
            for (int q = 0; q < ND_NW; ++q) t += s_warp[q][k];
            dst[k] = t;
        }
    }
    cluster.sync();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        v[k] = 0;
        for (int q = 0; q < C; ++q) v[k] += s_cl[turn][q][k];
    }
    turn ^= 1;
}

// Dot products of nv (1..4) basis vectors with u and w over the rows [i0, i1)
// of the CTA, by one warp: lane l ends with value l >> 1 of
// [vector][V^H u re, im, V^H w re, im].  8 rows per lane are summed as they
// come, those sums compensated.
template <class V>
__device__ __forceinline__ typename VT<V>::R sub_dots(const V* v0, int64_t ld, int nv, const V* su, const V* sw, int i0,
                                                      int i1, int lane) {
    using R = typename VT<V>::R;
    RowSum<R> acc[16];
    if constexpr (sizeof(R) == 8) {            // FP64: straight sums, 2 rows x 4 vectors in flight
        for (int i = i0 + lane; i < i1; i += 64) {
            V v[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int k = 0; k < 4; ++k) v[q][k] = (i + 32 * q < i1 && k < nv) ? v0[k * ld + i + 32 * q] : mk<V>(0, 0);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int e = i + 32 * q;
                const V u = e < i1 ? su[e] : mk<V>(0, 0), w = e < i1 ? sw[e] : mk<V>(0, 0);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    acc[4 * k].s = fma(v[q][k].x, u.x, fma(v[q][k].y, u.y, acc[4 * k].s));
                    acc[4 * k + 1].s = fma(v[q][k].x, u.y, fma(-v[q][k].y, u.x, acc[4 * k + 1].s));
                    acc[4 * k + 2].s = fma(v[q][k].x, w.x, fma(v[q][k].y, w.y, acc[4 * k + 2].s));
                    acc[4 * k + 3].s = fma(v[q][k].x, w.y, fma(-v[q][k].y, w.x, acc[4 * k + 3].s));
                }
            }
        }
    } else
    for (int i = i0 + lane; i < i1; i += 256) {
        R a[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) a[k] = 0;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {          // 4 rows x 4 vectors in flight
            V v[4][4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = i + (4 * h + q) * 32;
#pragma unroll
                for (int k = 0; k < 4; ++k) v[q][k] = (e < i1 && k < nv) ? v0[k * ld + e] : mk<V>(0, 0);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = i + (4 * h + q) * 32;
                const V u = e < i1 ? su[e] : mk<V>(0, 0), w = e < i1 ? sw[e] : mk<V>(0, 0);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    a[4 * k] = fma(v[q][k].x, u.x, fma(v[q][k].y, u.y, a[4 * k]));             // conj(v) * u
                    a[4 * k + 1] = fma(v[q][k].x, u.y, fma(-v[q][k].y, u.x, a[4 * k + 1]));
                    a[4 * k + 2] = fma(v[q][k].x, w.x, fma(v[q][k].y, w.y, a[4 * k + 2]));
                    a[4 * k + 3] = fma(v[q][k].x, w.y, fma(-v[q][k].y, w.x, a[4 * k + 3]));
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) acc[k].add(a[k]);
    }
    R t[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) t[k] = acc[k].s;
    return warp_sum_many<16>(t, lane);
}

template <bool GLOB, class V, class FW, class F>
__global__ void __launch_bounds__(ND_NT, 2)
k_subsolve(NdTables T, NdSizes z, NdMem mm, V* __restrict__ glob, const FW* __restrict__ fac, SubArgs<V, F> a,
           int keep_off, unsigned long long wait_ns, int stall, int* __restrict__ err) {
    namespace cg = cooperative_groups;
    using R = typename VT<V>::R;
    constexpr bool F64 = sizeof(V) == 16;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_abort, s_keep, s_task;
    __shared__ double s_red[ND_NW][3], s_sc[4];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)blockIdx.x, C = (int)gridDim.x, sub = (int)blockIdx.y;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    NdCta<V> nd;
    nd_enter<GLOB>(nd, T, z, mm, glob, smem, sub, rank, C, wait_ns, stall, &s_abort, err);
    cluster.sync();                            // the peers run before their shared memory is written
    const Sub S = a.subs[sub];
    const int m = a.m, rpr = sub_rows(S.n, C);
    const int64_t ra = S.off + min(S.n, (int64_t)rank * rpr), rb = S.off + min(S.n, (int64_t)(rank + 1) * rpr);
    const int nr = (int)(rb - ra);
    // the Krylov phases' shared memory, over the apply's vectors
    unsigned char* kp = smem + nd_layout<V>(z, mm.slt_smem, mm.u_glob, mm.y_glob).vec;
    double2* tot = reinterpret_cast<double2*>(kp);
    double2* hin = tot + 2 * m + 2;
    V* sc = reinterpret_cast<V*>(hin + m + 1);
    R* red = reinterpret_cast<R*>(sc + 2 * m + 2);
    V* s_uw = reinterpret_cast<V*>(reinterpret_cast<unsigned char*>(red) + ((size_t)(m / 4 + 2 + SUB_ITEMS) * 16 * sizeof(R) + 15) / 16 * 16);
    double2* part = a.partial + ((int64_t)sub * C) * (2 * m + 2);
    // rank 0: rotations and g of the cycle, kept in shared memory across the steps
    GivensArgs gl = a.g;
    gl.gv = reinterpret_cast<double2*>(smem + keep_off);
    gl.sn = gl.gv + m + 1;
    gl.pp = gl.sn + m;
    gl.pq = gl.pp + m + 1;
    gl.ip = gl.pq + m;
    double2* pre = gl.ip + 1;                  // [m + 1]
    double* target = reinterpret_cast<double*>(pre + m + 1);
    gl.cs = target + 2;
    gl.target = target;
    gl.Rm += (int64_t)sub * m * m;
    gl.active += sub; gl.kused += sub; gl.beta += sub;
    int turn = 0, total = 0, most = 0, steps = 0;
    unsigned long long w_dots = 0, w_upd = 0, n_apply = 0, n_res = 0;      // counted by thread 0 of rank 0

    for (int64_t r = ra + tid; r < rb; r += ND_NT) {
        a.x[r] = make_double2(0, 0);
        a.r[r] = a.b[r];
    }
    double bn = 0, prev = INFINITY;
    for (int cyc = 0; F64 || cyc < a.max_cycles; ++cyc) {
        double nn[2] = {0, 0};                 // ||r||^2, and of r rounded to the vector precision
        for (int64_t r = ra + tid; r < rb; r += ND_NT) {
            const double2 v = a.r[r];
            nn[0] = fma(v.x, v.x, fma(v.y, v.y, nn[0]));
            const double vx = (double)(R)v.x, vy = (double)(R)v.y;
            nn[1] = fma(vx, vx, fma(vy, vy, nn[1]));
        }
        if (tid == 0 && !nd.ok) nn[0] = nn[1] = NAN;      // a CTA's tables did not come: all of them stop
        cluster_sum<2>(nn, turn, rank, C);
        const double rn = sqrt(nn[0]), beta = sqrt(nn[1]);
        if (cyc == 0) bn = rn;
        // above the tolerance, and still falling (a residual that a cycle does
        // not halve has reached the accuracy that the arithmetic allows)
        if (!(rn > a.tol * bn && rn < 0.5 * prev && beta > 0)) break;
        prev = rn;
        if (F64 && total >= a.maxit) {
            if (rank == 0 && tid == 0) a.totals->no_conv = 1;
            break;
        }
        if (!F64) total = 0;
        const R ib = (R)(1.0 / beta);
        for (int64_t r = ra + tid; r < rb; r += ND_NT) {
            const double2 v = a.r[r];
            a.basis[r] = mk<V>((R)v.x * ib, (R)v.y * ib);
        }
        if (rank == 0 && tid == 0) {
            gl.gv[0] = make_double2(beta, 0);
            *target = F64 ? a.tol * bn : a.cycle_tol * beta;
        }
        cluster.sync();
        int j = 0;
        bool broke = false;
        double gp = 1, igp = 1;                // gamma of the previous step, and its inverse
        for (;; ++j) {
            const bool last = j == m || total >= a.maxit;
            V* uj = a.basis + (int64_t)j * a.n;
            V* zj = a.zbasis + (int64_t)j * a.n;
            V *su, *sw;
            if constexpr (GLOB) { su = uj + ra; sw = a.w + ra; }
            else { su = s_uw; sw = s_uw + rpr; }
            if (!last) {
                nd_apply_cta<GLOB>(nd, T, fac, uj, zj);
                cluster.sync();
            }
            // w = A z, and the products of u with itself and with w
            RowSum<R> cs[3];
            for (int i = tid; i < nr; i += ND_NT) {
                const V u = uj[ra + i];
                V w = mk<V>(0, 0);
                if (!last) w = sub_spmv<GLOB>(a, a.A, ra + i, zj, S.off);
                if (!GLOB) su[i] = u;
                sw[i] = w;
                cs[0].add(u.x * u.x + u.y * u.y);
                cs[1].add(u.x * w.x + u.y * w.y);
                cs[2].add(u.x * w.y - u.y * w.x);
            }
            {
                R c4[4] = {cs[0].s, 0, cs[1].s, cs[2].s};
                const R t = warp_sum_many<4>(c4, lane);
                if ((lane & 7) == 0 && lane != 8) s_red[warp][lane == 0 ? 0 : lane == 16 ? 1 : 2] = (double)t;
            }
            __syncthreads();
            // dot products: 4 basis vectors per warp, their rows in parts while there are few vectors
            const int ng = (j + 3) / 4;
            const int np = ng > 0 ? max(1, min((SUB_ITEMS + ng - 1) / ng, (nr + 127) / 128)) : 1;
            const int pr = ((nr + np - 1) / np + 31) / 32 * 32;
            for (int it = warp; it < ng * np; it += ND_NW) {
                const int g = it / np, p = it - g * np;
                const R t = sub_dots<V>(a.basis + (int64_t)(4 * g) * a.n + ra, a.n, min(4, j - 4 * g), su, sw, p * pr,
                                        min(nr, (p + 1) * pr), lane);
                if ((lane & 1) == 0) red[it * 16 + (lane >> 1)] = t;
            }
            __syncthreads();
            double2* mine = part + (int64_t)rank * (2 * m + 2);
            for (int k = tid; k < 2 * j + 2; k += ND_NT) {
                double2 t = make_double2(0, 0);
                if (k < 2 * j) {
                    const int v = k >> 1, o = (v & 3) * 4 + (k & 1) * 2;
                    for (int p = 0; p < np; ++p) {
                        t.x += (double)red[((v >> 2) * np + p) * 16 + o];
                        t.y += (double)red[((v >> 2) * np + p) * 16 + o + 1];
                    }
                } else if (k == 2 * j) {
                    for (int q = 0; q < ND_NW; ++q) t.x += s_red[q][0];
                } else {
                    for (int q = 0; q < ND_NW; ++q) { t.x += s_red[q][1]; t.y += s_red[q][2]; }
                }
                mine[k] = t;
            }
            cluster.sync();
            // totals and the scalar step, the same in every CTA
            for (int k = tid; k < 2 * j + 2; k += ND_NT) {
                double2 t[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    t[q] = q < C ? __ldcg(part + (int64_t)q * (2 * m + 2) + k) : make_double2(0, 0);
#pragma unroll
                for (int q = 1; q < 8; ++q)
                    if (q < C) t[0] = cadd(t[0], t[q]);
                tot[k] = t[0];
            }
            if (tid == 0) { s_task = 0; if (j == 0) s_keep = 1; }
            __syncthreads();
            // |s|^2 and s^H b.  FP64 instructions cost a warp 64 cycles whatever
            // its active lanes, so they run on as few warps as the columns need
            if (warp * 32 < j) {
                double v4[4] = {0, 0, 0, 0};
                for (int k = tid; k < j; k += ND_NT) {
                    const double2 sk = tot[2 * k], bk = tot[2 * k + 1];
                    v4[0] = fma(sk.x, sk.x, fma(sk.y, sk.y, v4[0]));
                    v4[1] = fma(sk.x, bk.x, fma(sk.y, bk.y, v4[1]));
                    v4[2] = fma(sk.x, bk.y, fma(-sk.y, bk.x, v4[2]));
                }
                const double t = warp_sum_many<4>(v4, lane);
                if ((lane & 7) == 0 && lane < 24) s_red[warp][lane >> 3] = t;
            }
            __syncthreads();
            if (warp == 0) {                   // gamma, 1 / gamma and d for everybody
                double ss = 0, sbr = 0, sbi = 0;
                for (int q = 0; q * 32 < min(j, ND_NT); ++q) { ss += s_red[q][0]; sbr += s_red[q][1]; sbi += s_red[q][2]; }
                const double c1 = tot[2 * j].x;
                const double2 c2 = tot[2 * j + 1];
                double gamma = 1.0, ig = 1.0;
                if (j > 0) {
                    const double g2 = c1 - ss;
                    ig = g2 > 0 ? rsqrt(g2) : INFINITY;
                    gamma = g2 > 0 ? g2 * ig : 0.0;      // 0: u_j lies in span(V) (a lucky breakdown)
                }
                if (lane == 0) {
                    s_sc[0] = isfinite(c1) && isfinite(c2.x) && isfinite(c2.y) && isfinite(gamma) ? gamma : -1.0;
                    s_sc[1] = ig;
                    s_sc[2] = (c2.x - sbr) * ig;
                    s_sc[3] = (c2.y - sbi) * ig;
                }
            }
            __syncthreads();
            const double gamma = s_sc[0];
            if (gamma < 0) {
                if (F64 && rank == 0 && tid == 0) a.totals->breakdown = 1;
                broke = true;
                break;                         // the totals are the same in every CTA: all of them leave here
            }
            const double ig = s_sc[1];
            {
                const double2 d = make_double2(s_sc[2], s_sc[3]);
                for (int k = tid; k < j; k += ND_NT) {
                    const double2 sk = tot[2 * k], bk = tot[2 * k + 1];
                    if (rank == 0) {
                        // Hessenberg column j-1: [b_{j-1}; d_{j-1}] + gamma_{j-1} s_j over gamma_{j-1} gamma_j
                        const double2 p = pre[k];
                        hin[k] = make_double2(p.x + gp * sk.x, p.y + gp * sk.y);
                        pre[k] = bk;
                    }
                    sc[k] = mk<V>((R)(-sk.x * ig), (R)(-sk.y * ig));
                    sc[j + k] = mk<V>((R)(-(bk.x - (sk.x * d.x - sk.y * d.y) * ig) * ig),
                                      (R)(-(bk.y - (sk.x * d.y + sk.y * d.x) * ig) * ig));
                }
                if (tid == ND_NT - 1) {
                    if (rank == 0) pre[j] = d;
                    sc[2 * j] = mk<V>((R)ig, (R)0);
                    sc[2 * j + 1] = mk<V>((R)(-d.x * ig * ig), (R)(-d.y * ig * ig));
                }
            }
            __syncthreads();
            if (rank == 0 && warp == 0 && j > 0) {     // the Givens step beside the update
                const bool keep = givens_core(gl, 0, j - 1, hin, gp * gamma, igp * ig, last);
                if (lane < C) *cluster.map_shared_rank(&s_keep, lane) = keep;
            }
            gp = gamma;
            igp = ig;
            if (!last) {
                // v_j over u_j and u_{j+1}: NU * 32 rows per warp and turn
                V* un = uj + a.n;
                const R cv = sc[2 * j].x, cur = sc[2 * j + 1].x, cui = sc[2 * j + 1].y;
                constexpr int NU = F64 ? 1 : 2;
                while (true) {
                    int t = 0;
                    if (lane == 0) t = atomicAdd(&s_task, 1);
                    t = __shfl_sync(0xffffffffu, t, 0);
                    if (t * 32 * NU >= nr) break;
                    V xo[NU], yo[NU];
                    int at[NU];
#pragma unroll
                    for (int q = 0; q < NU; ++q) {
                        at[q] = (t * NU + q) * 32 + lane;
                        if (at[q] >= nr) at[q] = -1;
                        const V u = at[q] >= 0 ? su[at[q]] : mk<V>(0, 0), w = at[q] >= 0 ? sw[at[q]] : mk<V>(0, 0);
                        xo[q] = mk<V>(cv * u.x, cv * u.y);
                        yo[q] = mk<V>(cv * w.x + cur * u.x - cui * u.y, cv * w.y + cur * u.y + cui * u.x);
                    }
                    constexpr int KB = 8;
                    const V* vb = a.basis + ra;
                    for (int k0 = 0; k0 < j; k0 += KB) {
                        V v[KB][NU];
#pragma unroll
                        for (int k = 0; k < KB; ++k)
#pragma unroll
                            for (int q = 0; q < NU; ++q)
                                v[k][q] = (k0 + k < j && at[q] >= 0) ? vb[(int64_t)(k0 + k) * a.n + at[q]] : mk<V>(0, 0);
#pragma unroll
                        for (int k = 0; k < KB; ++k) {
                            const int kk = min(k0 + k, j - 1);         // beyond j - 1 the vectors are zeros
                            const V al = sc[kk], be = sc[j + kk];
#pragma unroll
                            for (int q = 0; q < NU; ++q) {
                                xo[q].x = fma(al.x, v[k][q].x, fma(-al.y, v[k][q].y, xo[q].x));
                                xo[q].y = fma(al.x, v[k][q].y, fma(al.y, v[k][q].x, xo[q].y));
                                yo[q].x = fma(be.x, v[k][q].x, fma(-be.y, v[k][q].y, yo[q].x));
                                yo[q].y = fma(be.x, v[k][q].y, fma(be.y, v[k][q].x, yo[q].y));
                            }
                        }
                    }
#pragma unroll
                    for (int q = 0; q < NU; ++q)
                        if (at[q] >= 0) {
                            if (j > 0) uj[ra + at[q]] = xo[q];
                            un[ra + at[q]] = yo[q];
                        }
                }
                ++total;
                w_upd += (unsigned long long)(j + 2 + (j > 0 ? 2 : 1));
                ++n_apply;
            }
            w_dots += (unsigned long long)(j + 1 + (last ? 0 : 1));
            cluster.sync();
            if (!s_keep) break;
        }
        if (broke) break;
        // x += Z y, y = R^{-1} g over the j columns of the cycle
        steps += j;
        most = F64 ? steps : max(most, j);
        if (rank == 0 && warp == 0) backsolve(m, j, gl.Rm, gl.gv, tot, a.y + (int64_t)sub * m, lane);
        cluster.sync();
        for (int k = tid; k < j; k += ND_NT) {
            const double2 y = __ldcg(a.y + (int64_t)sub * m + k);
            sc[k] = mk<V>((R)y.x, (R)y.y);
        }
        __syncthreads();
        for (int64_t r0 = ra + tid; r0 < rb; r0 += 2 * ND_NT) {
            const bool two = r0 + ND_NT < rb;
            V s0 = mk<V>(0, 0), s1 = mk<V>(0, 0);
            constexpr int KB = F64 ? 4 : 8;
            for (int k0 = 0; k0 < j; k0 += KB) {
                V p[KB], q[KB];
#pragma unroll
                for (int k = 0; k < KB; ++k) {
                    const V* zk = a.zbasis + (int64_t)(k0 + k) * a.n + r0;
                    p[k] = k0 + k < j ? zk[0] : mk<V>(0, 0);
                    q[k] = (k0 + k < j && two) ? zk[ND_NT] : mk<V>(0, 0);
                }
#pragma unroll
                for (int k = 0; k < KB; ++k) {
                    const V y = sc[min(k0 + k, j - 1)];
                    s0.x = fma(y.x, p[k].x, fma(-y.y, p[k].y, s0.x));
                    s0.y = fma(y.x, p[k].y, fma(y.y, p[k].x, s0.y));
                    s1.x = fma(y.x, q[k].x, fma(-y.y, q[k].y, s1.x));
                    s1.y = fma(y.x, q[k].y, fma(y.y, q[k].x, s1.y));
                }
            }
            a.x[r0] = make_double2(a.x[r0].x + (double)s0.x, a.x[r0].y + (double)s0.y);
            if (two) a.x[r0 + ND_NT] = make_double2(a.x[r0 + ND_NT].x + (double)s1.x, a.x[r0 + ND_NT].y + (double)s1.y);
        }
        cluster.sync();
        // the FP64 residual
        for (int64_t r = ra + tid; r < rb; r += ND_NT) {
            const double2 t = sub_spmv<GLOB>(a, a.A64, r, a.x, S.off), b = a.b[r];
            a.r[r] = make_double2(b.x - t.x, b.y - t.y);
        }
        ++n_res;
    }
    if (rank == 0 && tid == 0) {
        atomicAdd(&a.totals->iters, (unsigned long long)steps);
        atomicAdd(&a.totals->dof_iters, (unsigned long long)steps * (unsigned long long)S.n);
        atomicMax(&a.totals->max_iters, most);
        const unsigned long long n = (unsigned long long)S.n;
        atomicAdd(a.kw, n_apply * n);
        atomicAdd(a.kw64, n_res * n);
        atomicAdd(a.kw + 1, w_dots * n * sizeof(V));
        atomicAdd(a.kw + 2, w_upd * n * sizeof(V));
        if (a.bt) {
            atomicAdd(a.bt, n_apply * (unsigned long long)T.welem[sub]);
            atomicAdd(a.bt + 1, n_apply * n);
        }
    }
}

}  // namespace thm
