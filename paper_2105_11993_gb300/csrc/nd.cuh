// Nested dissection of the subdomains: the elimination tree of P_i over the
// subdomain's cells and the tables that the factorisation (ndfactor.cu) and
// the solve (ndsolve.cuh) run from.  Built once per mesh (ndtree.cu).
//
// The cells of a subdomain are bisected recursively; a local DOF belongs to
// the smallest part of that recursion that holds all its cells, so a node's
// DOFs couple only to DOFs of its subtree and of its ancestors.  Order 2: the
// 4 bubbles of a cell are the DOFs of a leaf of their own.  The top
// log2(C) cuts form one root node (C: CTAs per subdomain); below it small
// nodes absorb their children, which trades a little arithmetic for depth.
//
// The order above knows the mesh only.  Where the elimination of a node is
// unstable with a system's coefficients, some of its unknowns move to an
// ancestor (ndfactor.cu): the trees of such subdomains are built again for that
// system with those moves, and their tables follow the mesh's (NdOwn).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <vector>

namespace thm {

constexpr int ND_NT = 256;                  // threads of a solve CTA
constexpr int ND_NW = ND_NT / 32;
constexpr uint32_t ND_NONE = 0xffffu;       // no child entry in a map half-word
constexpr uint32_t ND_NOROW = 0xffffffffu;  // padding row of a slice
constexpr size_t ND_SMEM_MAX = 226 * 1024; // dynamic; the kernels keep less than 1 KB of static shared memory
constexpr int ND_RESTART = 120;             // default restart length of the subdomain solves
constexpr uint32_t ND_U = 0x8000u;          // destination of a row: an entry of u (else of the vector)

// Tree node, as the factorisation sees it (nodes are sorted by depth, deepest first).
struct NdNode {
    int32_t s, b;             // eliminated unknowns, ancestor unknowns
    int32_t sub;
    int32_t child0, nchild;   // into the child list
    int32_t slt_f, slt_b;     // first forward resp. backward slice of its level (the root's rows: see its parts)
    int32_t row_f, row_b;     // first row within the level's forward resp. backward rows
    int32_t root_rows;        // root: rows per CTA; else 0
    int64_t rows0;            // local rows (s, then b; each part ascending) in the row list
    int64_t cmap0;            // the b unknowns' places in the parent's front
    int64_t front;            // offset of the (s+b)^2 front in its depth's workspace
};

// One depth of one CTA's subtrees (64 bytes; a CTA's levels are contiguous, deepest first, the root's last).
struct NdLev {
    int32_t v0, nv;           // vector entries of the level's nodes (each node padded to 4)
    int32_t nsf, sltf;        // forward slices: count, first (within the CTA's slice table)
    int32_t rowf, ymap;       // first forward row, first vector-entry map
    int32_t ksf;              // warps that share the columns of a forward slice
    int32_t nsb, sltb, rowb;  // backward slices
    int32_t idx;              // first index of the level's ancestor lists
    int32_t ksb;
    int32_t depth;
    int32_t pad[3];
};

struct NdPart {               // one CTA of one subdomain
    int32_t lev0, nlev;       // levels (the root's is number nlev)
    int32_t slt0, nslt;       // slice table
    int32_t nvec;             // vector: the root's unknowns, a zero entry, then the levels'
    int32_t sroot, rr0, nrr;  // root unknowns, and this CTA's share of them
    int32_t rmap0, pad;
    int64_t perm0;
};

struct NdTables {             // device tables
    const NdPart* parts;
    const NdLev* levs;
    const int2* slt;          // slices: {offset in the factor / 128, column quads}
    const uint32_t* rowd;     // rows: low half the staged-y offset (forward) or index list / 4 (backward), high half the destination
    const uint32_t* rowm;     // forward rows: children's u entries (mw words of two)
    const uint32_t* ymap;     // vector entries: the same
    const uint32_t* rmap;     // root unknowns: 2 mw words rank << 16 | entry, ~0 ends
    const uint16_t* idx;      // ancestor unknowns' vector entries
    const int32_t* perm;      // vector entry -> local row (-1: padding)
    const int64_t* welem;
    const struct Sub* subs;
    int32_t mw;
};

struct NdSizes {              // largest over the CTAs
    int32_t nlev = 0, nslt = 0, nvec = 0, ny = 0, nu[2] = {0, 0};
};

struct NdMove { int32_t row, node; };           // an unknown's node, where it is not the tree's choice
struct NdRef { int32_t sub, node, parent; };    // tree node (numbered within its subdomain's tree) of a node

struct NdHost {               // tables of a list of subdomains (the mesh's: of all)
    int C = 1, mw = 1;        // CTAs per subdomain; map words (of two children's entries)
    NdSizes z;
    int64_t fac_elems = 0;    // entries of a factor, with the padding of rows and slices
    std::vector<int64_t> welem;                 // per subdomain: values of the factor that a solve multiplies by
    std::vector<NdRef> node_ref;                // per node
    std::vector<int64_t> depth_node, depth_front;   // per depth, deepest first: first node (one more at the end), front entries
    std::vector<int32_t> depth_s, depth_n;      // largest s and s + b
    std::vector<NdPart> parts;
    std::vector<NdLev> levs;
    std::vector<int2> slt;
    std::vector<uint32_t> rowd, rowm, ymap, rmap;
    std::vector<uint16_t> idx;
    std::vector<int32_t> perm;
    std::vector<NdNode> nodes;
    std::vector<int32_t> rows, cmap, childs;
};

}  // namespace thm
