// The DDM-GMRES solve: block-preconditioned GMRES in every subdomain (Section
// 3.2, Eq. 7; subsolve.cuh), the impedance-trace exchange (Eqs. 5-6), GMRES on the
// interface system (Eq. 8), gluing, the FP64 true residual and iterative
// refinement.
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <string>

#include "kernels.cuh"
#include "krylov.cuh"
#include "ndsolve.cuh"
#include "solver.cuh"
#include "subsolve.cuh"

namespace thm {

__global__ void k_seg_reduce_real(int nseg, const int32_t* __restrict__ seg_ch, const double* __restrict__ part,
                                  double* __restrict__ out) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nseg) return;
    double acc = 0;
    for (int c = seg_ch[s]; c < seg_ch[s + 1]; ++c) acc += part[c];
    out[s] = acc;
}

// Start of a cycle: beta = ||r||, activity, g = (beta, 0, ...).  On the first
// cycle the per-segment target is tol * ||b_s|| (x = 0 there, so r = b).
// A segment whose true residual did not fall below half of its value at the
// previous cycle start has reached the accuracy its arithmetic allows
// (FP32 iterates: about cond(T_i) * 6e-8) and stops as well.
__global__ void k_cycle_start(int nseg, int m, const double* __restrict__ nrm2, double tol, int first,
                              double* __restrict__ target, double* __restrict__ beta, int* __restrict__ active,
                              int* __restrict__ kused, double2* __restrict__ gv, int* __restrict__ nact,
                              double* __restrict__ prev) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nseg) return;
    double b = sqrt(nrm2[s]);
    if (first) { target[s] = tol * b; prev[s] = INFINITY; }
    int a = b > target[s] && b > 0 && b < 0.5 * prev[s];
    prev[s] = b;
    active[s] = a;
    beta[s] = a ? b : 0.0;
    kused[s] = 0;
    for (int k = 0; k <= m; ++k) gv[(int64_t)s * (m + 1) + k] = make_double2(k == 0 && a ? b : 0.0, 0.0);
    if (a) atomicAdd(nact, 1);
}

// Second Gram-Schmidt update w -= V h2 with the per-chunk ||w||^2; the last
// block of each segment sums the segment's norm partials in chunk order and
// runs that segment's Givens step (so no separate reduction or Givens launch).
__global__ void __launch_bounds__(KT) k_update_givens(const Chunk* __restrict__ chunks, const double2* __restrict__ basis,
                                                      int64_t ld, int nk, double2* __restrict__ w,
                                                      double* __restrict__ nrm_part, const int* __restrict__ act,
                                                      GivensArgs ga, unsigned long long* __restrict__ work) {
    extern __shared__ double2 hk[];            // [nk] coefficients, then the Hessenberg column
    __shared__ double2 sa[KW * KSUB], sw[KSUB];
    __shared__ double s_n[KW], s_hn2;
    const Chunk c = chunks[blockIdx.x];
    if (act && !act[c.seg]) return;
    if (work && threadIdx.x == 0) atomicAdd(work, (unsigned long long)((nk + 2) * (c.end - c.begin) * sizeof(double2)));
    for (int k = threadIdx.x; k < nk; k += KT) hk[k] = ga.h2[(int64_t)c.seg * ga.ldh + k];
    __syncthreads();
    double nr = 0;
    for (int64_t e0 = c.begin; e0 < c.end; e0 += KSUB) {
        const double2 a = sub_chunk_update(basis, ld, nk, e0, c.end, hk, w, sa, sw);
        nr += a.x * a.x + a.y * a.y;
    }
    for (int o = 16; o > 0; o >>= 1) nr += __shfl_xor_sync(0xffffffffu, nr, o);
    if ((threadIdx.x & 31) == 0) s_n[threadIdx.x >> 5] = nr;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int q = 0; q < KSUB / 32; ++q) s += s_n[q];
        nrm_part[blockIdx.x] = s;
    }
    if (!last_block_of_segment(c.seg, ga.seg_ch, ga.cnt)) return;
    if (threadIdx.x < 32) {                    // the chunks' norms, lane by lane in chunk order
        double t = 0;
        for (int cc = ga.seg_ch[c.seg] + threadIdx.x; cc < ga.seg_ch[c.seg + 1]; cc += 32) t += __ldcg(&nrm_part[cc]);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) s_hn2 = t;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int j = ga.j;
        double2* hin = hk;                     // [j+1] h1 + h2
        for (int i = threadIdx.x; i <= j; i += 32)
            hin[i] = cadd(ga.h1[(int64_t)c.seg * ga.ldh + i], ga.h2[(int64_t)c.seg * ga.ldh + i]);
        __syncwarp();
        const double hn = sqrt(s_hn2);
        givens_core(ga, c.seg, j, hin, hn, 1.0 / hn);
    }
}

__global__ void __launch_bounds__(32) k_backsolve(int nseg, int m, const double2* __restrict__ Rm,
                                                  const double2* __restrict__ gv, const int* __restrict__ kused,
                                                  double2* __restrict__ y) {
    extern __shared__ double2 gsh[];           // [2m]
    const int s = blockIdx.x;
    if (s < nseg) backsolve(m, kused[s], Rm + (int64_t)s * m * m, gv + (int64_t)s * (m + 1), gsh, y + (int64_t)s * m, threadIdx.x);
}

// Right-hand side of every subdomain: sources + sum of received interface data.
__global__ void k_rhs(int64_t n, const double2* __restrict__ src, const int64_t* __restrict__ rowg_ptr,
                      const int32_t* __restrict__ rowg_idx, const double2* __restrict__ g, double2* __restrict__ b) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n) return;
    double2 v = src ? src[r] : make_double2(0, 0);
    if (g)
        for (int64_t p = rowg_ptr[r]; p < rowg_ptr[r + 1]; ++p) v = cadd(v, g[rowg_idx[p]]);
    b[r] = v;
}

// Impedance-trace exchange (Eq. 6):  G_{i<-j} = -G_{j<-i} + 2 i kappa omega (M_Sigma_ij u_j)[g],
// the face-mass product summed over the entry's terms (val already holds
// kappa*omega times the face mass, so that a batch of problems with different
// omega shares the kernel); (cr, ci) is the transmission coefficient in units
// of kappa*omega, (0, 1) for the impedance condition (i kappa omega), so the
// update is G = -G_partner + 2 (cr + i ci) (val . u_j).  A term on a Dirichlet
// DOF of u_j uses u_D when the sweep carries the Dirichlet lifting, else 0.
__global__ void k_exchange(int64_t n_if, const int32_t* __restrict__ partner, const int64_t* __restrict__ ptr,
                           const int32_t* __restrict__ tcol, const double* __restrict__ val, double cr, double ci,
                           const double2* __restrict__ g_in, const double2* __restrict__ u,
                           const double2* __restrict__ uD, double2* __restrict__ g_out) {
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n_if) return;
    double ar = 0, ai = 0;
    for (int64_t p = ptr[k]; p < ptr[k + 1]; ++p) {
        const int32_t c = tcol[p];
        double2 x = c >= 0 ? u[c] : (uD ? uD[-(int64_t)c - 1] : make_double2(0, 0));
        ar += val[p] * x.x;
        ai += val[p] * x.y;
    }
    double2 gp = g_in ? g_in[partner[k]] : make_double2(0, 0);
    g_out[k] = make_double2(-gp.x + 2.0 * (cr * ar - ci * ai), -gp.y + 2.0 * (cr * ai + ci * ar));
}

// u[d] += u_loc[owner(d)] on free DOFs
__global__ void k_glue_add(int64_t n_dof, const int32_t* __restrict__ owner, const double2* __restrict__ uloc,
                           double2* __restrict__ u) {
    int64_t d = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (d >= n_dof) return;
    int32_t o = owner[d];
    if (o >= 0) u[d] = cadd(u[d], uloc[o]);
}

__global__ void k_scatter_loc(int64_t n_loc, const int64_t* __restrict__ gdof, const double2* __restrict__ u,
                              double2* __restrict__ uloc) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r < n_loc) uloc[r] = u[gdof[r]];
}

// r_glob[d] = sum over the local copies of d of rl (free d), 0 on Dirichlet DOFs
__global__ void k_gather_sum(int64_t n_dof, const int64_t* __restrict__ cptr, const int32_t* __restrict__ cidx,
                             const double2* __restrict__ rl, double2* __restrict__ rg) {
    int64_t d = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (d >= n_dof) return;
    double2 a = make_double2(0, 0);
    for (int64_t p = cptr[d]; p < cptr[d + 1]; ++p) a = cadd(a, rl[cidx[p]]);
    rg[d] = a;
}

// owner split of a global vector into local sources
__global__ void k_owner_split(int64_t n_loc, const int64_t* __restrict__ gdof, const uint8_t* __restrict__ owner,
                              const double2* __restrict__ rg, double2* __restrict__ src) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r < n_loc) src[r] = owner[r] ? rg[gdof[r]] : make_double2(0, 0);
}

__global__ void k_norm2_blocks(int64_t n, const double2* __restrict__ x, double* __restrict__ part) {
    __shared__ double sw[32];
    double s = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double2 v = x[i];
        s += v.x * v.x + v.y * v.y;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += sw[q];
        part[blockIdx.x] = t;
    }
}

static inline unsigned nblk(int64_t n, int th = 256) { return (unsigned)((n + th - 1) / th); }

// ---------------------------------------------------------------------------
// Restarted GMRES on the interface system, one segment per problem: classical
// Gram-Schmidt with one full re-orthogonalisation (CGS2), Givens rotations in
// FP64.
// ---------------------------------------------------------------------------
struct KStats {
    int64_t iters = 0;       // sum over segments of Arnoldi steps
    int status = THM_OK;
};

struct Krylov {
    using V = double2;
    int64_t n = 0;
    int nseg = 0, m = 0, nch = 0;
    DArr<Chunk> d_chunks;
    DArr<int32_t> seg_ch;
    DArr<V> basis, w, r, t;
    DArr<double2> partial, h1, h2, Rm, sn, gv, pp, pq, ip, y;
    DArr<double> nrm_part, nrm, cs, beta, target, prev;
    DArr<int> active, kused, cnt;
    // monitor record of the latest Arnoldi step, 32 bytes: the active-segment
    // count, unused, the breakdown flag, then g_{j+1} of segment 0
    DArr<double2> mon;
    unsigned long long* work = nullptr;   // [2]: dot-product and update pass bytes (the system's counters), or null
    int* nact = nullptr;
    int* flag = nullptr;
    double2* gmon = nullptr;
    int* h_pinned = nullptr;
    std::vector<int> h_kused;
    double2* h_mon = nullptr;        // [2] the record of the latest step, pinned
    double h_beta0 = 0;              // ||r_0|| of segment 0 at the first cycle
    double last_rel = 1.0;           // latest residual estimate of segment 0, relative

    ~Krylov() {
        if (h_pinned) cudaFreeHost(h_pinned);
        if (h_mon) cudaFreeHost(h_mon);
    }

    void init(int64_t n_, int nseg_, int m_, const std::vector<Chunk>& chunks) {
        n = n_; nseg = nseg_; m = m_; nch = (int)chunks.size();
        d_chunks.upload(chunks);
        std::vector<int32_t> sc(nseg + 1, 0);
        for (const Chunk& c : chunks) sc[c.seg + 1]++;
        for (int s = 0; s < nseg; ++s) sc[s + 1] += sc[s];
        seg_ch.upload(sc);
        basis.alloc((size_t)(m + 1) * n);
        w.alloc(n); r.alloc(n); t.alloc(n);
        partial.alloc((size_t)nch * (2 * m + 2));
        h1.alloc((size_t)nseg * (m + 1)); h2.alloc((size_t)nseg * (m + 1));
        Rm.alloc((size_t)nseg * m * m);
        sn.alloc((size_t)nseg * m); cs.alloc((size_t)nseg * m);
        gv.alloc((size_t)nseg * (m + 1));
        pp.alloc((size_t)nseg * (m + 1)); pq.alloc((size_t)nseg * m); ip.alloc(nseg);
        y.alloc((size_t)nseg * m);
        nrm_part.alloc(nch); nrm.alloc(nseg); beta.alloc(nseg); target.alloc(nseg); prev.alloc(nseg);
        active.alloc(nseg); kused.alloc(nseg);
        cnt.alloc(nseg);
        cnt.zero(0);
        mon.alloc(2);
        mon.zero(0);
        nact = reinterpret_cast<int*>(mon.p);
        flag = nact + 2;
        gmon = mon.p + 1;
        if (!h_pinned) THM_CUDA(cudaMallocHost(&h_pinned, 2 * sizeof(int)));
        if (!h_mon) THM_CUDA(cudaMallocHost(&h_mon, 2 * sizeof(double2)));
        // the kernels are shared by every instance: only ever raise their limit
        // (coefficients and products of a step: 51 KB at the longest restart)
        const size_t dots_smem = 2 * (size_t)(m + 1) * sizeof(double2);
        THM_REQUIRE(m < 1600, "restart length too large");
        static size_t dots_attr = 0;
        if (dots_smem > dots_attr) {
            THM_CUDA(cudaFuncSetAttribute(k_chunk_dots, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dots_smem));
            THM_CUDA(cudaFuncSetAttribute(k_update_givens, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dots_smem));
            THM_CUDA(cudaFuncSetAttribute(k_update_dots, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dots_smem));
            THM_CUDA(cudaFuncSetAttribute(k_backsolve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dots_smem));
            dots_attr = dots_smem;
        }
        THM_CUDA(cudaDeviceSynchronize());
    }

    void seg_norm2(const V* x, cudaStream_t st) {
        THM_LAUNCH(THM_K_KRYLOV, st, k_chunk_norm2<V><<<nch, KT, 0, st>>>(d_chunks.p, x, nrm_part.p));
        THM_LAUNCH(THM_K_KRYLOV, st, k_seg_reduce_real<<<nblk(nseg), 256, 0, st>>>(nseg, seg_ch.p, nrm_part.p, nrm.p));
    }

    unsigned long long* kw(int k) const { return work ? work + k : nullptr; }

    int read_nact(cudaStream_t st) {
        THM_CUDA(cudaMemcpyAsync(h_pinned, nact, 2 * sizeof(int), cudaMemcpyDeviceToHost, st));
        THM_CUDA(cudaStreamSynchronize(st));
        return h_pinned[0];
    }

    // Solve A x = b for all segments, from x = 0.  A(in, out).
    KStats solve(const std::function<void(const V*, V*)>& A, const V* b, V* x, double tol, int maxit, cudaStream_t st) {
        KStats ks;
        int total = 0;
        bool first = true;
        THM_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), st));
        THM_CUDA(cudaMemsetAsync(x, 0, n * sizeof(V), st));
        THM_CUDA(cudaMemcpyAsync(r.p, b, n * sizeof(V), cudaMemcpyDeviceToDevice, st));
        while (true) {
            seg_norm2(r.p, st);
            THM_CUDA(cudaMemsetAsync(nact, 0, sizeof(int), st));
            THM_LAUNCH(THM_K_KRYLOV, st, k_cycle_start<<<nblk(nseg), 256, 0, st>>>(nseg, m, nrm.p, tol, first ? 1 : 0,
                                                      target.p, beta.p, active.p, kused.p, gv.p, nact, prev.p));
            if (first && nseg == 1) {
                double b0 = 0;
                THM_CUDA(cudaMemcpyAsync(&b0, beta.p, sizeof(double), cudaMemcpyDeviceToHost, st));
                THM_CUDA(cudaStreamSynchronize(st));
                h_beta0 = b0;
                last_rel = 1.0;
            }
            first = false;
            if (read_nact(st) == 0) break;
            if (total >= maxit) { ks.status = THM_ENOCONV; break; }
            THM_LAUNCH(THM_K_KRYLOV, st, k_chunk_scale<V><<<nch, 256, 0, st>>>(d_chunks.p, r.p, beta.p, basis.p, nullptr));
            // Waits for the record of the latest step; true when every segment has
            // stopped, or on a breakdown.  A step goes out only after this: one
            // beyond the last would run a whole sweep, on a basis vector that was
            // not written, to be thrown away (with the host three steps ahead 3 of
            // some 85 sweeps of a solve; the wait costs about 10 us a step).
            auto stopped = [&]() -> bool {
                THM_CUDA(cudaMemcpyAsync(h_mon, mon.p, 2 * sizeof(double2), cudaMemcpyDeviceToHost, st));
                THM_CUDA(cudaStreamSynchronize(st));
                const int* rec = reinterpret_cast<const int*>(h_mon);
                if (rec[2]) { ks.status = THM_EBREAKDOWN; return true; }
                if (nseg == 1 && h_beta0 > 0) last_rel = std::hypot(h_mon[1].x, h_mon[1].y) / h_beta0;
                return rec[0] == 0;
            };
            for (int j = 0; j < m && total < maxit; ++j) {
                V* vj = basis.p + (int64_t)j * n;
                A(vj, w.p);
                const int nk = j + 1;
                const size_t sm = (size_t)nk * sizeof(double2);
                // CGS2: h1 = V^H w, then w -= V h1 and h2 = V^H w in one pass, then
                // w -= V h2 (the dot kernels reduce their segments themselves); the
                // second update also forms ||w|| and the Givens step of each segment
                THM_LAUNCH(THM_K_DOTS, st, k_chunk_dots<<<nch, KT, sm, st>>>(d_chunks.p, basis.p, n, nk, w.p, partial.p, m + 1,
                                                                               active.p, seg_ch.p, cnt.p, h1.p, m + 1, nact,
                                                                               kw(0)));
                THM_LAUNCH(THM_K_UPDATE, st, k_update_dots<<<nch, KT, 2 * sm, st>>>(d_chunks.p, basis.p, n, nk, h1.p, m + 1, w.p,
                                                                                  partial.p, m + 1, active.p, seg_ch.p,
                                                                                  cnt.p, h2.p, kw(1)));
                GivensArgs ga{j, m, m + 1, h1.p, h2.p, Rm.p, cs.p, sn.p, gv.p, pp.p, pq.p, ip.p, target.p, active.p, kused.p, beta.p,
                              nact, flag, nseg == 1 ? gmon : nullptr, seg_ch.p, cnt.p};
                THM_LAUNCH(THM_K_UPDATE, st, k_update_givens<<<nch, KT, sm, st>>>(d_chunks.p, basis.p, n, nk, w.p, nrm_part.p,
                                                                                      active.p, ga, kw(1)));
                THM_LAUNCH(THM_K_KRYLOV, st, k_chunk_scale<V><<<nch, 256, 0, st>>>(d_chunks.p, w.p, beta.p, basis.p + (int64_t)(j + 1) * n, active.p));
                ++total;
                if (stopped()) break;
            }
            THM_CUDA(cudaGetLastError());
            // x += V y
            THM_LAUNCH(THM_K_KRYLOV, st, k_backsolve<<<nseg, 32, 2 * (size_t)m * sizeof(double2), st>>>(nseg, m, Rm.p, gv.p,
                                                                                                  kused.p, y.p));
            THM_LAUNCH(THM_K_KRYLOV, st, k_chunk_combine<V><<<nch, KT, (size_t)m * sizeof(double2), st>>>(d_chunks.p, basis.p, n, kused.p, y.p, m, t.p));
            THM_LAUNCH(THM_K_KRYLOV, st, k_axpy<V><<<nblk(n), 256, 0, st>>>(n, t.p, x));
            kused.download(h_kused, st);
            for (int s = 0; s < nseg; ++s) ks.iters += h_kused[s];
            if (ks.status == THM_EBREAKDOWN) break;
            A(x, w.p);
            THM_LAUNCH(THM_K_KRYLOV, st, k_sub<V><<<nblk(n), 256, 0, st>>>(n, b, w.p, r.p));
        }
        THM_CUDA(cudaGetLastError());
        return ks;
    }
};

// Workspace of the subdomain solves in one precision (k_subsolve).
template <class V>
struct SubWork {
    int m = 0;
    DArr<V> basis, zbasis, w;
    DArr<double2> partial, Rm, y;
    DArr<double> beta;
    DArr<int> active, kused, flag;
    void init(const thm_mesh* mesh, int m_) {
        THM_REQUIRE(m_ < (sizeof(V) == 8 ? 800 : 1600), "restart length too large");
        m = m_;
        const size_t n = mesh->n_loc, ns = mesh->n_sub;
        basis.alloc((size_t)(m + 1) * n);
        zbasis.alloc((size_t)m * n);
        w.alloc(n);
        partial.alloc(ns * mesh->nd.C * (2 * m + 2));
        Rm.alloc(ns * m * m);
        y.alloc(ns * m);
        beta.alloc(ns); active.alloc(ns); kused.alloc(ns); flag.alloc(1);
    }
};

// ---------------------------------------------------------------------------
struct Work {
    int m_in = 0, m_out = 0;
    bool has64 = false, has32 = false;
    SubWork<double2> in64;
    SubWork<float2> in32;
    Krylov outer;
    DArr<SolveTotals> totals;
    DArr<double2> b64, x64, r64, src, g0, gtmp, gb, gsol, uglob, uloc, rloc, rglob, ytmp;
    DArr<double> npart;
    // per-problem norms of global vectors (batches)
    DArr<double> pnpart, pnrm;
    DArr<int32_t> pseg_ch;
};

// The system's work counters (allocated and zeroed on first use).
static unsigned long long* kwork(const thm_sys* s) {
    if (!s->kwork.p) {
        s->kwork.alloc(8);
        s->kwork.zero(s->st);
    }
    return s->kwork.p;
}

static void ensure_work(thm_sys* s, bool fp32, int m_in, int m_out) {
    const thm_mesh* m = s->m;
    if (!s->w) s->w = new Work();
    Work* w = s->w;
    unsigned long long* kw = kwork(s);
    if (w->m_in != m_in) { w->has64 = w->has32 = false; w->m_in = m_in; }
    require_nd(m);
    if (!fp32 && !w->has64) {
        w->in64.init(m, m_in);
        w->has64 = true;
    }
    if (fp32 && !w->has32) {
        w->in32.init(m, m_in);
        w->has32 = true;
    }
    if (w->m_out != m_out && m->n_if > 0) {
        // one Krylov segment per problem (its contiguous range of interface
        // entries); a single problem is one segment over all of them
        std::vector<Chunk> oc;
        // chunks as small as a warp holds while there are SMs for them (152)
        const int64_t step = KSUB * std::max<int64_t>(1, (m->n_if + 152 * KSUB - 1) / (152 * KSUB));
        for (int p = 0; p < m->n_prob; ++p) {
            const int64_t b0 = m->n_prob > 1 ? m->prob_if_ptr[p] : 0;
            const int64_t b1 = m->n_prob > 1 ? m->prob_if_ptr[p + 1] : m->n_if;
            for (int64_t b = b0; b < b1; b += step) {
                Chunk c{};
                c.seg = p; c.begin = b; c.end = std::min<int64_t>(b1, b + step);
                oc.push_back(c);
            }
        }
        w->outer.init(m->n_if, m->n_prob, m_out, oc);
        w->m_out = m_out;
    }
    if (m->n_prob > 1 && w->pnrm.n == 0) {
        std::vector<int32_t> sc(m->n_prob + 1, 0);
        for (const Chunk& c : m->dof_chunks) sc[c.seg + 1]++;
        for (int p = 0; p < m->n_prob; ++p) sc[p + 1] += sc[p];
        w->pseg_ch.upload(sc);
        w->pnpart.alloc(std::max<size_t>(1, m->dof_chunks.size()));
        w->pnrm.alloc(m->n_prob);
    }
    if (w->b64.n == 0) {
        w->b64.alloc(m->n_loc); w->x64.alloc(m->n_loc); w->r64.alloc(m->n_loc); w->src.alloc(m->n_loc);
        w->totals.alloc(1);
        w->uloc.alloc(m->n_loc); w->rloc.alloc(m->n_loc); w->ytmp.alloc(m->n_loc);
        size_t ni = m->n_if > 0 ? m->n_if : 1;
        w->g0.alloc(ni); w->gtmp.alloc(ni); w->gb.alloc(ni); w->gsol.alloc(ni);
        w->uglob.alloc(m->n_dof); w->rglob.alloc(m->n_dof);
        w->npart.alloc(1024);
    }
    // the interface GMRES counts its Gram-Schmidt bytes as FP64
    w->outer.work = kw + 1;
    THM_CUDA(cudaMemsetAsync(w->totals.p, 0, sizeof(SolveTotals), s->st));
}



SolveCfg make_cfg(const thm_solve_opts* o) {
    SolveCfg c{};
    c.fp32 = o && o->mode == THM_MODE_MIXED;
    THM_REQUIRE(!o || o->mode == THM_MODE_FP64 || o->mode == THM_MODE_MIXED, "unknown mode");
    c.rtol = (o && o->rtol > 0) ? o->rtol : 1e-8;
    c.m_in = (o && o->inner_restart > 0) ? o->inner_restart : ND_RESTART;
    c.m_out = (o && o->outer_restart > 0) ? o->outer_restart : 600;
    c.inner_maxit = (o && o->inner_maxit > 0) ? o->inner_maxit : 2000;
    c.outer_maxit = (o && o->outer_maxit > 0) ? o->outer_maxit : 2000;
    c.max_refine = (o && o->max_refine > 0) ? o->max_refine : 6;
    c.inner_tol = (o && o->inner_tol > 0) ? o->inner_tol : 1e-11;
    c.cycle_tol = 1e-5;
    c.relax = o ? o->relax : 0;
    c.outer_method = o ? o->outer_method : THM_OUTER_GMRES;
    THM_REQUIRE(c.outer_method == THM_OUTER_GMRES || c.outer_method == THM_OUTER_JACOBI, "unknown outer method");
    c.precond = o ? o->precond : THM_PRECOND_BLOCKDIAG;
    THM_REQUIRE(c.precond == THM_PRECOND_BLOCKDIAG || c.precond == THM_PRECOND_FULL, "unknown preconditioner");
    if (const char* e = getenv("THM_CYCLE_TOL")) c.cycle_tol = atof(e);
    c.outer_tol = (o && o->outer_tol > 0) ? o->outer_tol : 1e-9;
    return c;
}

// The SELL face-term arrays of a precision (3-D only; 2-D keeps them diagonal).
static inline void bv_arrays(const thm_sys* s, const double*, const double** g, const double** sg) {
    *g = s->m->dim == 3 ? s->bvg64.p : nullptr;
    *sg = s->m->dim == 3 ? s->bvs64.p : nullptr;
}
static inline void bv_arrays(const thm_sys* s, const float*, const float** g, const float** sg) {
    *g = s->m->dim == 3 ? s->bvg32.p : nullptr;
    *sg = s->m->dim == 3 ? s->bvs32.p : nullptr;
}

template <class V, class F>
static void apply_T(const thm_sys* s, const F* val, const F* bg, const F* bs, int use_bs, const V* x, V* y) {
    const thm_mesh* m = s->m;
    const F *bvg, *bvs;
    bv_arrays(s, val, &bvg, &bvs);
    unsigned long long* work = kwork(s) + (sizeof(F) == 4 ? 4 : 0);      // rows processed
    if (m->col16)
        THM_LAUNCH(THM_K_SPMV, s->st,
                   (k_spmv<V, F, uint16_t><<<nblk(m->n_loc), 256, 0, s->st>>>(
                       m->n_loc, m->d_slice_ptr.p, m->d_sell_col16.p, m->d_subs.p, SpmvMat<F>{val, bg, bs, bvg, bvs},
                       use_bs, x, y,
                       m->d_loc_sub.p, work)));
    else
        THM_LAUNCH(THM_K_SPMV, s->st,
                   (k_spmv<V, F, int32_t><<<nblk(m->n_loc), 256, 0, s->st>>>(
                       m->n_loc, m->d_slice_ptr.p, m->d_sell_col.p, m->d_subs.p, SpmvMat<F>{val, bg, bs, bvg, bvs},
                       use_bs, x, y,
                       m->d_loc_sub.p, work)));
}

// The block preconditioner of every subdomain: one cluster of nd.C CTAs each.
// Two CTAs to an SM where their vectors fit (each hides the other's barriers
// and L2 latency); what outgrows shared memory (nd_fit) is in a workspace of
// the system.  False: it does not fit.
template <class V, class FW>
static bool nd_memory(const thm_sys* s, bool glob, size_t more, size_t keep, NdMem* out, size_t* keep_off, size_t* smem) {
    const thm_mesh* m = s->m;
    require_nd(m);
    const NdSizes& z = s->nd_sizes(NdCplx<FW>::value);
    if (!s->bt_work.p) {
        s->bt_work.alloc(4);
        s->bt_work.zero(s->st);
    }
    NdMem mm{};
    // L2 prefetch of the factor two levels ahead of its use where all factors
    // together are more than a small part of L2 (129 MB), which the bases of
    // the solves share: FP32 sweeps with 80 to 140 MB of factors 18.1 -> 17.0 ms
    // (64 cubes of 8^3 cells) and 26.6 -> 25.6 ms (64 squares of 32^2, order 2);
    // factors of a few MB are in L2 anyway, and asking costs 1% (4 squares of
    // 24^2, order 2: 641 -> 648 ms a solve).
    mm.prefetch = m->nd.fac_elems * (int64_t)sizeof(FW) >= (int64_t)16 << 20;
    // THM_BT_CPL_GLOBAL=1 runs everything from global memory that can be there
    const char* force = getenv("THM_BT_CPL_GLOBAL");
    *smem = nd_fit<V>(z, glob, more, keep, &mm, force && atoi(force) != 0);
    if (*smem == 0) return false;
    const size_t entries = (size_t)(mm.glob_stride * m->n_sub * m->nd.C);
    if (s->nd_glob.n < entries) s->nd_glob.alloc(entries);
    *out = mm;
    *keep_off = *smem - keep;
    return true;
}

// The wait for a solve kernel's table copies gives up after
// THM_BT_WAIT_LIMIT_MS (default 1000 ms); THM_TEST_STALL_TMA=1 holds the
// copies back, so that a test can see the bounded wait expire and
// THM_ETIMEOUT come back.
static unsigned long long nd_wait_ns() {
    const char* lim = getenv("THM_BT_WAIT_LIMIT_MS");
    return 1000000ull * (unsigned long long)(lim ? std::max(1, atoi(lim)) : 1000);
}
static int nd_stall() {
    const char* stall = getenv("THM_TEST_STALL_TMA");
    return stall && atoi(stall) != 0;
}

// Launches a solve kernel, one cluster of nd.C CTAs per subdomain.
template <class... P, class... A>
static void nd_launch(const thm_sys* s, int cls, void (*kernel)(P...), size_t smem, A... args) {
    const thm_mesh* m = s->m;
    THM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ND_SMEM_MAX));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(m->nd.C, m->n_sub);
    cfg.blockDim = dim3(ND_NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s->st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = m->nd.C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    THM_LAUNCH(cls, s->st, THM_CUDA(cudaLaunchKernelEx(&cfg, kernel, P(args)...)));
}

template <class V, class FW>
static void nd_apply(const thm_sys* s, const FW* fac, const V* x, V* y) {
    size_t smem = 0, keep_off = 0;
    NdMem mm{};
    const bool glob = !nd_memory<V, FW>(s, false, 0, 0, &mm, &keep_off, &smem);
    THM_REQUIRE(!glob || (nd_memory<V, FW>(s, true, 0, 0, &mm, &keep_off, &smem)),
                "subdomain too large for the shared-memory block solve");
    // the work counter follows the Eq. 7 (real-factor) applies only
    unsigned long long* work = NdCplx<FW>::value ? nullptr : s->bt_work.p + (sizeof(FW) == 4 ? 2 : 0);
    nd_launch(s, THM_K_PINV, glob ? k_nd_solve<true, V, FW> : k_nd_solve<false, V, FW>, smem, nd_tables(s, NdCplx<FW>::value), s->nd_sizes(NdCplx<FW>::value), mm, reinterpret_cast<V*>(s->nd_glob.p),
              fac, nd_wait_ns(), nd_stall(), s->dev_err.p, work, x, y);
}

// The solve totals counted on the device since prepare (or the last call).
static void collect(thm_sys* s, RunStats& rs) {
    SolveTotals t;
    THM_CUDA(cudaMemcpyAsync(&t, s->w->totals.p, sizeof(t), cudaMemcpyDeviceToHost, s->st));
    THM_CUDA(cudaStreamSynchronize(s->st));
    THM_CUDA(cudaMemsetAsync(s->w->totals.p, 0, sizeof(t), s->st));
    rs.inner += (int64_t)t.iters;
    rs.dof_iters += (int64_t)t.dof_iters;
    rs.max_inner = std::max(rs.max_inner, t.max_iters);
    if (t.no_conv && rs.status == THM_OK) rs.status = THM_ENOCONV;
    if (t.breakdown && rs.status == THM_OK) rs.status = THM_EBREAKDOWN;
}

template <class V, class FW, class F>
static void subsolve(thm_sys* s, const SolveCfg& c, SubWork<V>& k, const FW* fac, const F* val, const F* bg, const F* bs,
                     const double2* b, double2* x) {
    const thm_mesh* m = s->m;
    Work* w = s->w;
    int64_t nmax = 0;
    for (const auto& S : m->subs) nmax = std::max(nmax, S.n);
    const int rows = sub_rows(nmax, m->nd.C);
    size_t smem = 0, keep_off = 0;
    NdMem mm{};
    // glob: u and w of the rows stay in global memory, like the apply's vectors
    // as need be.  A restart length whose scalars outgrow shared memory (about
    // 1,000; less where the vectors fill it) is cut to what fits: such a cycle
    // restarts there.
    int mr = k.m;
    bool glob = false;
    while (true) {
        const size_t keep = sub_keep_bytes(mr);
        glob = !m->col16 || !nd_memory<V, FW>(s, false, sub_krylov_bytes<V>(rows, mr, 0), keep, &mm, &keep_off, &smem);
        if (!glob || nd_memory<V, FW>(s, true, sub_krylov_bytes<V>(rows, mr, 1), keep, &mm, &keep_off, &smem)) break;
        THM_REQUIRE(mr > 8, "subdomain too large for the shared-memory block solve");
        mr -= 8;
    }
    SubArgs<V, F> a{};
    const bool f32 = sizeof(F) == 4;
    a.m = mr;
    a.maxit = f32 ? mr : c.inner_maxit;
    a.max_cycles = std::max(1, c.inner_maxit / std::max(1, c.m_in));
    a.tol = c.inner_tol;
    a.cycle_tol = c.cycle_tol;
    a.col16 = m->col16;
    a.n = m->n_loc;
    a.b = b; a.x = x; a.r = w->r64.p;
    a.basis = k.basis.p; a.zbasis = k.zbasis.p; a.w = k.w.p;
    a.partial = k.partial.p; a.y = k.y.p;
    a.g = GivensArgs{0, mr, mr + 1, nullptr, nullptr, k.Rm.p, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, k.active.p, k.kused.p,
                     k.beta.p, nullptr, k.flag.p, nullptr, nullptr, nullptr};
    a.subs = m->d_subs.p;
    a.slice_ptr = m->d_slice_ptr.p;
    a.col = m->d_sell_col.p;
    a.col_rel = m->d_sell_col16.p;
    a.A.val = val; a.A.bg = bg; a.A.bs = bs;
    bv_arrays(s, val, &a.A.bvg, &a.A.bvs);
    a.A64.val = s->val64.p; a.A64.bg = s->bg64.p; a.A64.bs = s->bs64.p;
    bv_arrays(s, a.A64.val, &a.A64.bvg, &a.A64.bvs);
    a.totals = w->totals.p;
    a.kw64 = kwork(s);
    a.kw = a.kw64 + (f32 ? 4 : 0);
    a.bt = NdCplx<FW>::value ? nullptr : s->bt_work.p + (f32 ? 2 : 0);
    nd_launch(s, THM_K_SUBSOLVE, glob ? k_subsolve<true, V, FW, F> : k_subsolve<false, V, FW, F>, smem, nd_tables(s, NdCplx<FW>::value), s->nd_sizes(NdCplx<FW>::value), mm, reinterpret_cast<V*>(s->nd_glob.p),
              fac, a, (int)keep_off, nd_wait_ns(), nd_stall(), s->dev_err.p);
}

// Solve all subdomain problems T_i x_i = b_i (b, x FP64 local vectors).  Each
// mixed cycle runs to cycle_tol relative to its own right-hand side (the FP32
// limit), also when the refined solve needs less: with the relaxed interface
// tolerances the margin is what keeps the interface GMRES from stalling (a
// floor at a quarter of the subdomain tolerance took 937 interface steps
// against 362 on the 256x256 order-2 workload, measured).
static void subdomain_solves(thm_sys* s, const SolveCfg& c, const double2* b, double2* x) {
    Work* w = s->w;
    const bool full = c.precond == THM_PRECOND_FULL;
    if (c.fp32) {
        if (full) subsolve<float2, float2, float>(s, c, w->in32, s->facc32.p, s->val32.p, s->bg32.p, s->bs32.p, b, x);
        else subsolve<float2, float, float>(s, c, w->in32, s->fac32.p, s->val32.p, s->bg32.p, s->bs32.p, b, x);
    } else {
        if (full) subsolve<double2, double2, double>(s, c, w->in64, s->facc64.p, s->val64.p, s->bg64.p, s->bs64.p, b, x);
        else subsolve<double2, double, double>(s, c, w->in64, s->fac64.p, s->val64.p, s->bg64.p, s->bs64.p, b, x);
    }
}

// One sweep: x = T^{-1}(src + R g_in), g_out = exchange(g_in, x).
static void sweep(thm_sys* s, const SolveCfg& c, const double2* src, const double2* g_in, double2* g_out,
                  double2* x, RunStats& rs, const double2* uD = nullptr) {
    const thm_mesh* m = s->m;
    Work* w = s->w;
    cudaStream_t st = s->st;
    THM_LAUNCH(THM_K_DDM, st, k_rhs<<<nblk(m->n_loc), 256, 0, st>>>(m->n_loc, src, m->d_rowg_ptr.p, m->d_rowg_idx.p,
                                          m->n_if > 0 ? g_in : nullptr, w->b64.p));
    subdomain_solves(s, c, w->b64.p, x);
    if (m->n_if > 0 && g_out)
        THM_LAUNCH(THM_K_DDM, st, k_exchange<<<nblk(m->n_if), 256, 0, st>>>(m->n_if, m->d_if_partner.p, m->d_if_ptr.p,
                                                                           m->d_if_tcol.p, s->if_val.p,
                                                                           s->trans_re, s->trans_im, g_in, x, uD,
                                                                           g_out));
    rs.sweeps++;
    THM_CUDA(cudaGetLastError());
}

static double global_norm(thm_sys* s, const double2* x, int64_t n);

// DDM solve of Eq. 8 for local sources src -> local solution uloc.
static void ddm_solve(thm_sys* s, const SolveCfg& c, const double2* src, double2* uloc, RunStats& rs,
                      const double2* uD) {
    const thm_mesh* m = s->m;
    Work* w = s->w;
    cudaStream_t st = s->st;
    if (m->n_if == 0) {
        sweep(s, c, src, nullptr, nullptr, uloc, rs);
        return;
    }
    // b = A_src(0): sweep with sources and zero interface data
    w->g0.zero(st);
    sweep(s, c, src, w->g0.p, w->gb.p, uloc, rs, uD);
    if (c.outer_method == THM_OUTER_JACOBI) {
        // fixed point of g = A_src(g) = A g + b (the plain iteration of Eq. 8):
        // g_{k+1} = A_src(g_k) from g_1 = b, stopped on ||g_k - A_src(g_k)|| <= tol ||b||
        const double bn = global_norm(s, w->gb.p, m->n_if);
        double2* g = w->gb.p;
        double2* gn = w->gsol.p;
        int k = 0;
        bool conv = bn == 0;
        while (!conv && k < c.outer_maxit) {
            sweep(s, c, src, g, gn, uloc, rs, uD);
            THM_LAUNCH(THM_K_KRYLOV, st, k_sub<double2><<<nblk(m->n_if), 256, 0, st>>>(m->n_if, g, gn, w->gtmp.p));
            const double r = global_norm(s, w->gtmp.p, m->n_if);
            ++k;
            if (r <= c.outer_tol * bn) conv = true;
            else std::swap(g, gn);
        }
        rs.outer += k;
        if (!conv && rs.status == THM_OK) rs.status = THM_ENOCONV;
        sweep(s, c, src, g, nullptr, uloc, rs, uD);
        return;
    }
    auto A = [&](const double2* v, double2* out) {
        SolveCfg cr = c;
        if (c.relax) {
            // inexact Krylov: GMRES tolerates matvec errors of about
            // tol / ||r_k|| (relative), so the subdomain solves may loosen as
            // the outer residual falls.  The subdomain residual only bounds
            // the sweep error up to a constant, hence the safety factor
            // 1e-2 and the ceiling 1e-6 (looser settings stall the outer
            // iteration).
            const double eta = 1e-2 * c.outer_tol / std::max(w->outer.last_rel, 1e-300);
            cr.inner_tol = std::min(1e-6, std::max(c.inner_tol, eta));
        }
        sweep(s, cr, nullptr, v, w->gtmp.p, w->ytmp.p, rs);
        THM_LAUNCH(THM_K_KRYLOV, st, k_sub<double2><<<nblk(m->n_if), 256, 0, st>>>(m->n_if, v, w->gtmp.p, out));   // (I - A) v
    };
    static const bool verbose = getenv("THM_VERBOSE") != nullptr;
    std::function<void(const double2*, double2*)> Av = A;
    if (verbose) {
        Av = [&, t0 = std::chrono::steady_clock::now()](const double2* v, double2* out) {
            int64_t before = rs.inner;
            A(v, out);
            collect(s, rs);
            double el = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
            fprintf(stderr, "[thm] sweep %d: inner %lld (max %d) t=%.3fs\n", rs.sweeps,
                    (long long)(rs.inner - before), rs.max_inner, el);
        };
    }
    KStats ko = w->outer.solve(Av, w->gb.p, w->gsol.p, c.outer_tol, c.outer_maxit, st);
    rs.outer += (int)ko.iters;
    if (ko.status != THM_OK && rs.status == THM_OK) rs.status = ko.status;
    sweep(s, c, src, w->gsol.p, nullptr, uloc, rs, uD);
}

static double global_norm(thm_sys* s, const double2* x, int64_t n) {
    Work* w = s->w;
    const int nb = 512;
    THM_LAUNCH(THM_K_DDM, 0, k_norm2_blocks<<<nb, 256, 0, s->st>>>(n, x, w->npart.p));
    std::vector<double> h(nb);
    THM_CUDA(cudaMemcpyAsync(h.data(), w->npart.p, nb * sizeof(double), cudaMemcpyDeviceToHost, s->st));
    THM_CUDA(cudaStreamSynchronize(s->st));
    double t = 0;
    for (double v : h) t += v;
    return std::sqrt(t);
}

// Per-problem 2-norms of a global vector (a batch of independent problems:
// each owns a contiguous range of global DOFs), deterministic order.
static std::vector<double> problem_norms(thm_sys* s, const double2* x) {
    const thm_mesh* m = s->m;
    Work* w = s->w;
    std::vector<double> h(m->n_prob, 0.0);
    const int nch = (int)m->dof_chunks.size();
    if (nch > 0) {
        THM_LAUNCH(THM_K_DDM, s->st, k_chunk_norm2<double2><<<nch, KT, 0, s->st>>>(m->d_dof_chunks.p, x, w->pnpart.p));
        THM_LAUNCH(THM_K_DDM, s->st, k_seg_reduce_real<<<nblk(m->n_prob), 256, 0, s->st>>>(m->n_prob, w->pseg_ch.p,
                                                                                          w->pnpart.p, w->pnrm.p));
        THM_CUDA(cudaMemcpyAsync(h.data(), w->pnrm.p, m->n_prob * sizeof(double), cudaMemcpyDeviceToHost, s->st));
        THM_CUDA(cudaStreamSynchronize(s->st));
    }
    for (double& v : h) v = std::sqrt(v);
    return h;
}

// The largest relative residual over the problems (r_p / f_p; a problem with
// f_p = 0 has u_p = 0 exactly and counts as converged).
static double max_relative(const std::vector<double>& rn, const std::vector<double>& fn) {
    double r = 0;
    for (size_t p = 0; p < rn.size(); ++p)
        if (fn[p] > 0) r = std::max(r, rn[p] / fn[p]);
    return r;
}

// A bounded device-side wait that gave up leaves a flag: report THM_ETIMEOUT.
static void check_device_error(thm_sys* s) {
    int h = 0;
    THM_CUDA(cudaMemcpyAsync(&h, s->dev_err.p, sizeof(int), cudaMemcpyDeviceToHost, s->st));
    THM_CUDA(cudaStreamSynchronize(s->st));
    if (h) {
        THM_CUDA(cudaMemsetAsync(s->dev_err.p, 0, sizeof(int), s->st));
        fail(THM_ETIMEOUT, "a bounded wait for the table copies of a solve kernel gave up");
    }
}

// FP64 true residual r = f - K u for a local right-hand-side split f_loc of f.
static double true_residual_rhs(thm_sys* s, const double2* f_loc, const double2* u, double2* rglob) {
    const thm_mesh* m = s->m;
    Work* w = s->w;
    cudaStream_t st = s->st;
    THM_LAUNCH(THM_K_DDM, st, k_scatter_loc<<<nblk(m->n_loc), 256, 0, st>>>(m->n_loc, m->d_loc_gdof.p, u, w->uloc.p));
    apply_T<double2, double>(s, s->kloc_val64(), s->bg64.p, s->bs64.p, 0, w->uloc.p, w->ytmp.p);   // K^loc
    THM_LAUNCH(THM_K_DDM, st, k_sub<double2><<<nblk(m->n_loc), 256, 0, st>>>(m->n_loc, f_loc, w->ytmp.p, w->rloc.p));
    THM_LAUNCH(THM_K_DDM, st, k_gather_sum<<<nblk(m->n_dof), 256, 0, st>>>(m->n_dof, m->d_copy_ptr.p, m->d_copy_idx.p, w->rloc.p, rglob));
    return global_norm(s, rglob, m->n_dof);
}

// Refined DDM solve of K_FF u_F = f, u initialised with u0 on all DOFs (the
// Dirichlet values, or zeros).  f_res is the local split of f (summed over
// copies it is f); f_src the sources of the first DDM solve, which differ from
// f_res by the transmission terms of u0 on Dirichlet DOFs of Sigma.
int solve_rhs(thm_sys* s, const SolveCfg& c, const double2* f_src, const double2* f_loc, const double2* u0,
              double2* u, RunStats& rs, double& rel) {
    const thm_mesh* m = s->m;
    Work* w = s->w;
    cudaStream_t st = s->st;
    THM_LAUNCH(THM_K_DDM, st, k_gather_sum<<<nblk(m->n_dof), 256, 0, st>>>(m->n_dof, m->d_copy_ptr.p, m->d_copy_idx.p, f_loc, w->rglob.p));
    const bool batch = m->n_prob > 1;
    std::vector<double> fnp;
    double fn;
    if (batch) {
        fnp = problem_norms(s, w->rglob.p);
        fn = 0;
        for (double v : fnp) fn = std::max(fn, v);
    } else {
        fn = global_norm(s, w->rglob.p, m->n_dof);
    }
    if (u0) THM_CUDA(cudaMemcpyAsync(u, u0, m->n_dof * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    else THM_CUDA(cudaMemsetAsync(u, 0, m->n_dof * sizeof(double2), st));
    if (!std::isfinite(fn)) {                    // a non-finite right-hand side (Dirichlet data or sources)
        THM_CUDA(cudaStreamSynchronize(st));
        rel = fn;
        rs.status = THM_EBREAKDOWN;
        return THM_EBREAKDOWN;
    }
    THM_CUDA(cudaMemcpyAsync(w->src.p, f_src, m->n_loc * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    rel = fn > 0 ? 1.0 : 0.0;
    for (int it = 0; it < c.max_refine && fn > 0; ++it) {
        // the first DDM solve carries the Dirichlet lifting (u0 = u_D); the
        // refinement corrections have zero Dirichlet values
        ddm_solve(s, c, w->src.p, w->x64.p, rs, it == 0 ? u0 : nullptr);
        rs.refine++;
        THM_LAUNCH(THM_K_DDM, st, k_glue_add<<<nblk(m->n_dof), 256, 0, st>>>(m->n_dof, m->d_owner_loc.p, w->x64.p, u));
        double rn = true_residual_rhs(s, f_loc, u, w->rglob.p);
        rel = batch ? max_relative(problem_norms(s, w->rglob.p), fnp) : rn / fn;
        if (!std::isfinite(rel)) { rs.status = THM_EBREAKDOWN; break; }
        if (rel <= c.rtol) break;
        THM_LAUNCH(THM_K_DDM, st, k_owner_split<<<nblk(m->n_loc), 256, 0, st>>>(m->n_loc, m->d_loc_gdof.p, m->d_loc_is_owner.p,
                                                                               w->rglob.p, w->src.p));
    }
    collect(s, rs);
    THM_CUDA(cudaGetLastError());
    check_device_error(s);
    if (rs.status == THM_EBREAKDOWN) return THM_EBREAKDOWN;
    if (rel > c.rtol) return THM_ENOCONV;
    return THM_OK;
}

void fill_stats(const RunStats& rs, double rel, double sec, thm_stats* stats) {
    if (!stats) return;
    stats->outer_iters = rs.outer;
    stats->sweeps = rs.sweeps;
    stats->refine_steps = rs.refine;
    stats->inner_iters = rs.inner;
    stats->dof_iters = rs.dof_iters;
    stats->max_inner_iters = rs.max_inner;
    stats->rel_residual = rel;
    stats->seconds = sec;
}

void prepare(thm_sys* s, const SolveCfg& c) {
    ensure_factor(s, c.fp32);
    if (c.precond == THM_PRECOND_FULL) ensure_factor_full(s, c.fp32);
    ensure_work(s, c.fp32, c.m_in, c.m_out);
}

int solve(thm_sys* s, const thm_solve_opts* opts, double2* u, thm_stats* stats) {
    auto t0 = std::chrono::steady_clock::now();
    SolveCfg c = make_cfg(opts);
    prepare(s, c);
    RunStats rs;
    double rel = 0;
    int rc = solve_rhs(s, c, s->f_loc.p, s->f_res.p, s->uD.p, u, rs, rel);
    double sec = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    fill_stats(rs, rel, sec, stats);
    return rc;
}

// ---- diagnostics -----------------------------------------------------------
void apply_local(thm_sys* s, int op, int mode, const double2* x, double2* y) {
    bool f32 = mode == THM_MODE_MIXED;
    THM_REQUIRE(op == THM_OP_T || op == THM_OP_PINV || op == THM_OP_KLOC || op == THM_OP_TINV, "unknown op");
    if (op == THM_OP_PINV || op == THM_OP_TINV) {
        ensure_factor(s, f32);
        if (op == THM_OP_TINV) {
            ensure_factor_full(s, f32);
            if (f32) nd_apply<double2, float2>(s, s->facc32.p, x, y);
            else nd_apply<double2, double2>(s, s->facc64.p, x, y);
        } else {
            if (f32) nd_apply<double2, float>(s, s->fac32.p, x, y);
            else nd_apply<double2, double>(s, s->fac64.p, x, y);
        }
        THM_CUDA(cudaStreamSynchronize(s->st));
        check_device_error(s);
    } else {
        int use_bs = op == THM_OP_T;
        if (f32) apply_T<double2, float>(s, use_bs ? s->val32.p : s->kloc_val32(), s->bg32.p, s->bs32.p, use_bs, x, y);
        else apply_T<double2, double>(s, use_bs ? s->val64.p : s->kloc_val64(), s->bg64.p, s->bs64.p, use_bs, x, y);
    }
    THM_CUDA(cudaGetLastError());
    THM_CUDA(cudaStreamSynchronize(s->st));
}

int sweep_diag(thm_sys* s, const thm_solve_opts* opts, int with_sources, const double2* g_in, double2* g_out,
               double2* uloc, thm_stats* stats) {
    SolveCfg c = make_cfg(opts);
    prepare(s, c);
    RunStats rs;
    sweep(s, c, with_sources ? s->f_loc.p : nullptr, g_in, g_out, uloc, rs, with_sources ? s->uD.p : nullptr);
    collect(s, rs);
    check_device_error(s);
    if (stats) {
        memset(stats, 0, sizeof(*stats));
        stats->sweeps = rs.sweeps;
        stats->inner_iters = rs.inner;
        stats->dof_iters = rs.dof_iters;
        stats->max_inner_iters = rs.max_inner;
    }
    return rs.status;
}

}  // namespace thm

thm_sys::~thm_sys() { delete w; }
