// Internal structures of the THM DDM-GMRES library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <cstring>
#include <memory>
#include <string>
#include <vector>

#include "nd.cuh"
#include "thm.h"

namespace thm {

struct Error {
    int code;
    std::string msg;
};

[[noreturn]] void fail(int code, const std::string& msg);
void set_last_error(const std::string& msg);

#define THM_CUDA(call)                                                                 \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess)                                                         \
            ::thm::fail(e_ == cudaErrorMemoryAllocation ? THM_ENOMEM : THM_ECUDA,      \
                        std::string(#call) + ": " + cudaGetErrorString(e_));           \
    } while (0)

#define THM_REQUIRE(cond, msg)                                                         \
    do {                                                                               \
        if (!(cond)) ::thm::fail(THM_EINVAL, msg);                                     \
    } while (0)

// Owning device array.
template <class T>
struct DArr {
    T* p = nullptr;
    size_t n = 0;
    DArr() = default;
    DArr(const DArr&) = delete;
    DArr& operator=(const DArr&) = delete;
    ~DArr() { release(); }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
    }
    void alloc(size_t count) {
        release();
        n = count;
        if (count) THM_CUDA(cudaMalloc(&p, count * sizeof(T)));
    }
    void zero(cudaStream_t st) {
        if (n) THM_CUDA(cudaMemsetAsync(p, 0, n * sizeof(T), st));
    }
    void upload(const std::vector<T>& h, cudaStream_t st = 0) {
        alloc(h.size());
        if (n) THM_CUDA(cudaMemcpyAsync(p, h.data(), n * sizeof(T), cudaMemcpyHostToDevice, st));
    }
    void download(std::vector<T>& h, cudaStream_t st = 0) const {
        h.resize(n);
        if (n) {
            THM_CUDA(cudaMemcpyAsync(h.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost, st));
            THM_CUDA(cudaStreamSynchronize(st));
        }
    }
};

void prof_begin(int cls, cudaStream_t st);
void prof_end(int cls, cudaStream_t st);
void prof_set(unsigned mask);
void prof_read(int cls, int64_t* launches, double* ms);

// Every kernel launch of the library goes through THM_LAUNCH (launch count,
// optional CUDA-event timing of its class).
#define THM_LAUNCH(cls, st, ...)            \
    do {                                    \
        ::thm::prof_begin((cls), (st));     \
        __VA_ARGS__;                        \
        ::thm::prof_end((cls), (st));       \
    } while (0)

// Device copies of elimination-tree tables (nd.cuh).
struct NdDev {
    DArr<NdPart> parts;
    DArr<NdLev> levs;
    DArr<int2> slt;
    DArr<uint32_t> rowd, rowm, ymap, rmap;
    DArr<uint16_t> idx;
    DArr<int32_t> perm, rows, cmap, childs;
    DArr<int64_t> welem;
    DArr<NdNode> nodes;
};

// Lengths of the arrays that tables are put behind.  place_tables: moves their
// positions there; false if one outgrows 32 bits.
struct NdPlace { size_t levs, slt, rowd, ymap, rmap, idx, perm, fac; };

// Tables of a system that moved unknowns up the trees of some subdomains: the
// mesh's tables followed by those of these subdomains, which `parts` points to.
// (nodes, rows, cmap, childs: of the subdomains eliminated last.)
struct NdOwn {
    NdDev d;
    NdSizes z;                // of both
    int64_t fac_elems = 0;
    std::vector<NdPart> parts;
    std::vector<int64_t> welem;
    std::vector<std::vector<NdMove>> moves;     // [n_sub]
};

constexpr int SELL_C = 32;       // rows per SELL slice (one warp)
constexpr int CHUNK = 1024;      // elements per reduction chunk of a segment

struct Sub {
    int64_t off;      // first local row
    int64_t n;        // free DOFs
    int64_t ne;       // free edge DOFs (rows off .. off+ne-1); cell bubbles follow
};

// A contiguous piece of one segment, used for deterministic segmented reductions.
struct Chunk {
    int32_t seg;
    int32_t pad;
    int64_t begin;
    int64_t end;
};

}  // namespace thm

struct thm_mesh {
    int dim = 0, order = 0, dpc = 0, epc = 0, max_block = 0;
    int64_t n_vert = 0, n_cell = 0, n_bface = 0, n_edge = 0, n_dof = 0;
    int n_sub = 0;
    std::vector<double> coords;
    std::vector<int64_t> cells;
    std::vector<int32_t> cell_sub;
    std::vector<int64_t> bfaces;
    std::vector<uint8_t> btag;
    std::vector<int64_t> edge_lo, edge_hi;          // sorted (lo, hi)
    std::vector<int64_t> cell_dofs;                 // [n_cell][dpc]
    std::vector<int8_t> cell_signs;                 // [n_cell][dpc]
    std::vector<uint8_t> is_dir;                    // [n_dof]
    std::vector<int64_t> dir_edges;                 // edges carrying Dirichlet DOFs
    std::vector<int64_t> dir_dofs;                  // Dirichlet DOFs, increasing
    thm::DArr<int64_t> d_dir_dofs;

    // local (per-subdomain, free DOFs) structure
    int64_t n_loc = 0;
    std::vector<thm::Sub> subs;
    std::vector<int64_t> loc_gdof;                  // [n_loc]
    std::vector<int32_t> loc_sub;                   // [n_loc]
    std::vector<int32_t> cell_loc;                  // [n_cell][dpc] local row or -1
    // SELL-32 pattern of P_i (all subdomains), columns are local indices
    int64_t n_slices = 0, n_slots = 0;
    std::vector<int64_t> slice_ptr;                 // [n_slices+1]
    std::vector<int32_t> sell_col;                  // [n_slots]; padding = own row
    // the same columns relative to the row's subdomain (col - off of the
    // row's subdomain) in 16 bits, for the SpMV, when every subdomain has at
    // most 65,536 local DOFs (col16); the factorisation keeps sell_col
    std::vector<uint16_t> sell_col16;
    bool col16 = false;
    std::vector<uint8_t> sell_pad;                  // [n_slots] 1 = padding
    // assembly plan: cells holding each local row (ascending), <= maxc
    int maxc = 0;
    std::vector<int32_t> row_cell, row_k;           // [n_loc][maxc]
    // faces with impedance (kind 1, Gamma^inf) or transmission (kind 2, Sigma)
    // terms; fd DOFs per face (2-D order 1: 1, order 2: 2, 3-D: 4)
    static constexpr int RF = 4;                     // faces per local row, at most
    int fd = 0;
    int64_t n_face = 0;
    std::vector<int32_t> face_v;                    // [n_face][4] vertices, face-local tensor order
    std::vector<int32_t> face_dof;                  // [n_face][fd]
    std::vector<int8_t> face_sgn;                   // [n_face][fd]
    std::vector<int8_t> face_kind;                  // [n_face]
    std::vector<int32_t> face_sub;                  // [n_face][2] subdomains (-1: none)
    std::vector<int32_t> face_loc;                  // [n_face][2][fd] local rows per side (-1: Dirichlet)
    std::vector<int32_t> row_face;                  // [n_loc][RF] face ids (-1: none)
    std::vector<int8_t> row_face_a, row_face_side;  // [n_loc][RF]
    // elimination trees of the subdomains (the block preconditioner's factorisation)
    thm::NdHost nd;
    bool nd_ok = false;                             // false: a subdomain outgrows the solve kernel
    thm::NdDev ndd;
    // interface entries (directed pairs i <- j, one per free DOF on Sigma_ij)
    int64_t n_if = 0;
    std::vector<int32_t> if_recv, if_send, if_rowi, if_partner;
    std::vector<int64_t> if_gdof;
    // terms of (M_Sigma_ij u_j)[g] per entry: face, a, b, sender column (-(gdof+1): Dirichlet)
    std::vector<int64_t> if_ptr;
    std::vector<int32_t> if_tf, if_tcol;
    std::vector<int8_t> if_ta, if_tb;
    std::vector<int64_t> rowg_ptr;                  // [n_loc+1] local row -> entries received
    std::vector<int32_t> rowg_idx;
    // independent problems sharing the mesh (a batch): subdomain -> problem,
    // each problem's contiguous range of global DOFs and of interface entries,
    // and reduction chunks over the global DOFs segmented by problem
    int n_prob = 1;
    mutable bool assembled = false;                 // a system was built on this mesh
    std::vector<int32_t> sub_prob;                  // [n_sub]
    std::vector<int64_t> prob_dof_ptr, prob_if_ptr; // [n_prob+1]
    std::vector<thm::Chunk> dof_chunks;
    // global <-> local
    std::vector<int32_t> owner_loc;                 // [n_dof] lowest-subdomain copy, -1 Dirichlet
    std::vector<int64_t> copy_ptr;                  // [n_dof+1]
    std::vector<int32_t> copy_idx;
    std::vector<uint8_t> loc_is_owner;              // [n_loc]

    // device mirrors
    thm::DArr<double> d_coords;
    thm::DArr<int32_t> d_cells, d_cell_dofs, d_cell_loc, d_sell_col, d_row_cell, d_row_k;
    thm::DArr<uint16_t> d_sell_col16;
    thm::DArr<int64_t> d_edge_lo, d_edge_hi, d_slice_ptr, d_dir_edges, d_loc_gdof, d_rowg_ptr,
        d_copy_ptr;
    thm::DArr<int8_t> d_cell_signs, d_face_sgn, d_face_kind, d_row_face_a, d_row_face_side, d_if_ta, d_if_tb;
    thm::DArr<uint8_t> d_sell_pad, d_loc_is_owner;
    thm::DArr<int32_t> d_if_rowi, d_if_partner, d_rowg_idx, d_owner_loc, d_copy_idx, d_loc_sub, d_face_v,
        d_face_dof, d_face_loc, d_row_face, d_if_tf, d_if_tcol;
    thm::DArr<int64_t> d_if_ptr;
    thm::DArr<thm::Sub> d_subs;
    thm::DArr<thm::Chunk> d_dof_chunks;
};

namespace thm { struct Work; }

// Assembled system of one (mesh, mu^{-1}, omega, kappa, E^inc).
struct thm_sys {
    const thm_mesh* m = nullptr;
    cudaStream_t st = 0;
    double omega = 0, kappa = 0;       // omega: the first problem's (the only one unless batched)
    std::vector<double> omega_prob;    // [n_prob]
    thm::DArr<double> w2c;             // [n_cell] omega^2 of the cell's problem
    thm::DArr<double> kwf;             // [n_face] kappa*omega of the face's problem
    thm::DArr<double> omd;             // [n_dir_edges] omega of the Dirichlet edge's problem
    double pol[6] = {0};   // complex [dim]
    double dir[3] = {0};
    thm::DArr<double> mu_inv;          // [n_cell]
    thm::DArr<double> ref;             // reference matrices (see assemble.cu)
    thm::DArr<double> val64;           // SELL values of P_i = Re(T_i), FP64
    thm::DArr<float> val32;            // same, FP32
    // transmission coefficient on Sigma_ij in units of kappa*omega: (0, 1) is
    // i kappa omega, the impedance condition of Eq. 5; a real part adds
    // trans_re * kappa omega M_Sigma to Re(T_i) (and then K_i^loc, which has no
    // Sigma terms, gets value arrays of its own)
    double trans_re = 0.0, trans_im = 1.0;
    thm::DArr<double> valK64;          // SELL values of Re(K_i^loc) when trans_re != 0
    thm::DArr<float> valK32;
    const double* kloc_val64() const { return valK64.p ? valK64.p : val64.p; }
    const float* kloc_val32() const { return valK32.p ? valK32.p : val32.p; }
    thm::DArr<double> eps;             // [n_cell] relative permittivity (mass-term weight), 1 if not given
    thm::DArr<double> bg64, bs64;      // kappa*omega * diagonal face masses: Gamma^inf, Sigma
    thm::DArr<float> bg32, bs32;
    thm::DArr<double> if_val;          // values of the interface-entry terms (face masses)
    thm::DArr<double> bvg64, bvs64;    // 3-D: kappa*omega face masses on the SELL pattern (Gamma^inf, Sigma)
    thm::DArr<float> bvg32, bvs32;
    thm::DArr<double2> uD;             // [n_dof] Dirichlet values
    // Dirichlet values given by the caller (thm_assemble_dirichlet) instead of
    // the moments of a plane wave: [n_dir] in increasing global-DOF order
    bool dir_user = false;
    thm::DArr<double2> dir_vals;
    thm::DArr<double2> f_loc;          // [n_loc] subdomain sources: -(T_i)_{F,D} u_D (Eq. 5)
    thm::DArr<double2> f_res;          // [n_loc] split of the global right-hand side: -(K_i^loc)_{F,D} u_D
    // factors of P_i over the elimination trees (lazily built per precision)
    bool fac64_ok = false, fac32_ok = false;
    thm::DArr<double> fac64;
    thm::DArr<float> fac32;
    // complex factors of the full 2x2 block operator (Section 3.2's
    // alternative preconditioner), lazily built per precision
    bool facc64_ok = false, facc32_ok = false;
    thm::DArr<double2> facc64;
    thm::DArr<float2> facc32;
    // tables of the factors of P_i and of T_i where they are not the mesh's (else null)
    std::unique_ptr<thm::NdOwn> own, ownc;
    const thm::NdSizes& nd_sizes(bool cplx) const {
        const auto& o = cplx ? ownc : own;
        return o ? o->z : m->nd.z;
    }
    thm::DArr<int> dev_err;            // set by a device-side bounded wait that gave up
    // workspace of the solve kernel for subdomains whose vectors outgrow shared memory
    mutable thm::DArr<double2> nd_glob;
    // block-solve work actually done, per factor precision ([0..1] FP64, [2..3]
    // FP32): values read and local rows processed, summed by the kernel over
    // the subdomains it did not skip
    mutable thm::DArr<unsigned long long> bt_work;
    // work counters of the SpMV and Gram-Schmidt kernels, [8]: (FP32 ? 4 : 0)
    // + 0 SpMV rows processed, 1 dot-product pass bytes, 2 update pass bytes
    mutable thm::DArr<unsigned long long> kwork;
    // solver workspace (allocated on first solve, see solve.cu)
    thm::Work* w = nullptr;
    ~thm_sys();
};

namespace thm {
void build_mesh(thm_mesh* m);
void build_nd(thm_mesh* m);
void require_nd(const thm_mesh* m);
// Tables of the listed subdomains for 2^p CTAs each; moves: per subdomain of
// the mesh, or null.  False: an index outgrows its 16 bits, or a CTA's vectors
// its shared memory.
bool build_tables(const thm_mesh* m, NdHost& H, const std::vector<int>& list, int p,
                  const std::vector<std::vector<NdMove>>* moves);
bool place_tables(NdHost& H, const NdPlace& at);
NdSizes larger(NdSizes a, const NdSizes& b);
NdTables nd_tables(const thm_sys* s, bool cplx);
void assemble(thm_sys* s);
void ensure_factor(thm_sys* s, bool fp32);
void ensure_factor_full(thm_sys* s, bool fp32);
}  // namespace thm
