// Assembly of the subdomain operators T_i = P_i + i B_i (Section 2, the
// integrals (A), (M), (B) and Eq. 3; Section 3.1, the transmission term of
// Eq. 5), the Dirichlet data and the lifting.
#include <cmath>

#include "common.cuh"
#include "element.cuh"

namespace thm {

// ---------------------------------------------------------------------------
// Reference matrices.  Every component of a reference basis function (and of
// its curl) is c * f(xi) * g(eta) with f, g from five quadratics; integrals of
// products of two such terms are exact sums of monomial integrals 1/(i+j+1).
// Output layout: ref[0] = int curl_i curl_j, ref[1] = int phi_i,x phi_j,x,
// ref[2] = int phi_i,y phi_j,y on the unit square (12 x 12 each, row-major).
// Per cell of sides a (xi) and b (eta):  A = ref0/(ab),  M = (b/a) ref1 + (a/b) ref2.
// ---------------------------------------------------------------------------
__constant__ double c_poly[5][3] = {
    {1, 0, 0},     // 1
    {0, 1, 0},     // t
    {1, -1, 0},    // 1 - t
    {0, 1, -1},    // q(t)  = t (1 - t)
    {1, -2, 0},    // q'(t) = 1 - 2t
};

struct Term {
    double c;
    int f, g, h;      // 1-D factors in xi, eta, zeta (h = 0: the constant, for 2-D)
};

// Terms (x component, y component, curl) of the 12 order-2 functions in the
// local order [W0 G0 W1 G1 W2 G2 W3 G3 B0 B1 B2 B3]; order 1 uses W0..W3.
__device__ void basis_terms(int order, int i, Term& x, Term& y, Term& cu) {
    const Term Z{0, 0, 0, 0};
    // Whitney functions of local edges 0..3
    const Term Wx[4] = {{1, 0, 2}, {1, 0, 1}, Z, Z};
    const Term Wy[4] = {Z, Z, {1, 2, 0}, {1, 1, 0}};
    const Term Wc[4] = {{1, 0, 0}, {-1, 0, 0}, {-1, 0, 0}, {1, 0, 0}};
    // gradient functions grad(q(s) * ramp)
    const Term Gx[4] = {{1, 4, 2}, {1, 4, 1}, {-1, 0, 3}, {1, 0, 3}};
    const Term Gy[4] = {{-1, 3, 0}, {1, 3, 0}, {1, 2, 4}, {1, 1, 4}};
    // cell bubbles
    const Term Bx[4] = {{1, 2, 3}, {1, 1, 3}, Z, Z};
    const Term By[4] = {Z, Z, {1, 3, 2}, {1, 3, 1}};
    const Term Bc[4] = {{-1, 2, 4}, {-1, 1, 4}, {1, 4, 2}, {1, 4, 1}};
    if (order == 1) {
        x = Wx[i]; y = Wy[i]; cu = Wc[i];
        return;
    }
    if (i < 8) {
        int k = i >> 1;
        if ((i & 1) == 0) { x = Wx[k]; y = Wy[k]; cu = Wc[k]; }
        else { x = Gx[k]; y = Gy[k]; cu = Z; }
    } else {
        int k = i - 8;
        x = Bx[k]; y = By[k]; cu = Bc[k];
    }
}

__device__ double int1(int f, int g) {
    double s = 0;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            if (c_poly[f][i] != 0 && c_poly[g][j] != 0) s += c_poly[f][i] * c_poly[g][j] / (double)(i + j + 1);
    return s;
}

__device__ double int2(const Term& a, const Term& b) {
    if (a.c == 0 || b.c == 0) return 0.0;
    return a.c * b.c * int1(a.f, b.f) * int1(a.g, b.g) * int1(a.h, b.h);
}

// Order-1 hex: 12 Whitney functions in the local edge order (xi-edges at
// (eta,zeta) = 00,10,01,11, then eta-edges at (xi,zeta), then zeta-edges at
// (xi,eta)); comp[3] = value components, cu[3] = reference curl components.
// L(t;0) = 1 - t (poly 2), L(t;1) = t (poly 1), dL(0) = -1, dL(1) = +1.
__device__ void basis_terms3(int i, Term* comp, Term* cu) {
    const Term Z{0, 0, 0, 0};
    const int ax = i / 4, e0 = (i % 4) & 1, e1 = (i % 4) >> 1;
    const int L0 = e0 ? 1 : 2, L1 = e1 ? 1 : 2;
    const double d0 = e0 ? 1.0 : -1.0, d1 = e1 ? 1.0 : -1.0;
    for (int k = 0; k < 3; ++k) { comp[k] = Z; cu[k] = Z; }
    if (ax == 0) {           // (L(eta) L(zeta), 0, 0); curl = (0, L(eta) dL(zeta), -dL(eta) L(zeta))
        comp[0] = Term{1, 0, L0, L1};
        cu[1] = Term{d1, 0, L0, 0};
        cu[2] = Term{-d0, 0, 0, L1};
    } else if (ax == 1) {    // (0, L(xi) L(zeta), 0); curl = (-L(xi) dL(zeta), 0, dL(xi) L(zeta))
        comp[1] = Term{1, L0, 0, L1};
        cu[0] = Term{-d1, L0, 0, 0};
        cu[2] = Term{d0, 0, 0, L1};
    } else {                 // (0, 0, L(xi) L(eta)); curl = (L(xi) dL(eta), -dL(xi) L(eta), 0)
        comp[2] = Term{1, L0, L1, 0};
        cu[0] = Term{d1, L0, 0, 0};
        cu[1] = Term{-d0, 0, L1, 0};
    }
}

// ref layout (144 doubles per matrix, row stride nb):
//  2-D: [0] int curl curl, [1] int phi_x phi_x, [2] int phi_y phi_y,
//       [6] face (edge) scalars: [0] int 1*1, [1] int q'(s)^2
//  3-D: [0..2] int curl_a curl_a (a = xi, eta, zeta), [3..5] int phi_a phi_a,
//       [6], [7] the order-1 quad face mass parts (row stride 4)
__global__ void k_ref_matrices(int dim, int order, int nb, double* ref) {
    for (int t = threadIdx.x; t < nb * nb; t += blockDim.x) {
        int i = t / nb, j = t % nb;
        if (j < i) continue;
        if (dim == 2) {
            Term xi, yi, ci, xj, yj, cj;
            basis_terms(order, i, xi, yi, ci);
            basis_terms(order, j, xj, yj, cj);
            double a = int2(ci, cj), mx = int2(xi, xj), my = int2(yi, yj);
            ref[0 * 144 + i * nb + j] = a;  ref[0 * 144 + j * nb + i] = a;
            ref[1 * 144 + i * nb + j] = mx; ref[1 * 144 + j * nb + i] = mx;
            ref[2 * 144 + i * nb + j] = my; ref[2 * 144 + j * nb + i] = my;
        } else {
            Term vi[3], ci[3], vj[3], cj[3];
            basis_terms3(i, vi, ci);
            basis_terms3(j, vj, cj);
            for (int k = 0; k < 3; ++k) {
                double aa = int2(ci[k], cj[k]), mm = int2(vi[k], vj[k]);
                ref[k * 144 + i * nb + j] = aa;       ref[k * 144 + j * nb + i] = aa;
                ref[(3 + k) * 144 + i * nb + j] = mm; ref[(3 + k) * 144 + j * nb + i] = mm;
            }
        }
    }
    if (threadIdx.x == 0) {
        if (dim == 2) {
            ref[6 * 144 + 0] = int1(0, 0);
            ref[6 * 144 + 1] = int1(4, 4);
        } else {
            for (int i = 0; i < 4; ++i)
                for (int j = 0; j < 4; ++j) {
                    Term xi, yi, ci, xj, yj, cj;
                    basis_terms(1, i, xi, yi, ci);
                    basis_terms(1, j, xj, yj, cj);
                    ref[6 * 144 + i * 4 + j] = int2(xi, xj);
                    ref[7 * 144 + i * 4 + j] = int2(yi, yj);
                }
        }
    }
}

// Gather-by-row assembly of P_i in the SELL layout.  Entry (r, col) sums the
// cells holding both DOFs in ascending cell order; entry (col, r) visits the
// same cells in the same order with exactly symmetric reference entries, so
// P_i is bit-symmetric.
__global__ void k_assemble(int dim, int64_t n_loc, int nb, int maxc, const double* __restrict__ ref,
                           const double* __restrict__ X, const int32_t* __restrict__ cells,
                           const int8_t* __restrict__ signs, const int32_t* __restrict__ cell_loc,
                           const double* __restrict__ mu, const double* __restrict__ w2c,
                           const int64_t* __restrict__ slice_ptr, const int32_t* __restrict__ col,
                           const uint8_t* __restrict__ pad, const int32_t* __restrict__ row_cell,
                           const int32_t* __restrict__ row_k, double* __restrict__ val64,
                           float* __restrict__ val32) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n_loc) return;
    int64_t sl = r / SELL_C;
    int lane = (int)(r % SELL_C);
    int64_t base = slice_ptr[sl];
    int w = (int)((slice_ptr[sl + 1] - base) / SELL_C);
    for (int t = 0; t < w; ++t) {
        int64_t idx = base + (int64_t)t * SELL_C + lane;
        double v = 0.0;
        if (!pad[idx]) {
            int32_t cc = col[idx];
            for (int u = 0; u < maxc; ++u) {
                int32_t c = row_cell[r * maxc + u];
                if (c < 0) break;
                int kr = row_k[r * maxc + u];
                for (int kc = 0; kc < nb; ++kc) {
                    if (cell_loc[(int64_t)c * nb + kc] != cc) continue;
                    double hh[3];
                    cell_sides(X, dim, cells, c, hh);
                    double s = (double)(signs[(int64_t)c * nb + kr] * signs[(int64_t)c * nb + kc]);
                    v += s * cell_entry(dim, ref, nb, mu[c], w2c[c], hh, kr, kc);
                }
            }
        }
        val64[idx] = v;
        val32[idx] = (float)v;
    }
}

// Impedance / transmission face terms, gathered per local row from the faces
// whose terms reach it (kind 1: Gamma^inf, kind 2: Sigma), times kappa*omega.
// 2-D: the face mass is diagonal, stored per row (bg, bs).  3-D: the face mass
// couples the four edges of a face; stored on the SELL pattern (bvg, bvs).
__global__ void k_face_terms(int dim, int64_t n_loc, int fd, const double* __restrict__ ref,
                             const double* __restrict__ X, const int32_t* __restrict__ face_v,
                             const int8_t* __restrict__ face_sgn, const int8_t* __restrict__ face_kind,
                             const int32_t* __restrict__ face_loc, const int32_t* __restrict__ row_face,
                             const int8_t* __restrict__ row_face_a, const int8_t* __restrict__ row_face_side,
                             const int64_t* __restrict__ slice_ptr, const int32_t* __restrict__ col,
                             const uint8_t* __restrict__ pad, const double* __restrict__ kwf, double tre,
                             double tim, double* val64, float* val32, double* bg64,
                             double* bs64, float* bg32,
                             float* bs32, double* bvg64, double* bvs64, float* bvg32, float* bvs32) {
    // Sigma terms: (tre + i tim) kappa omega M_Sigma; the imaginary part goes to
    // the face-term arrays, a real part (tre != 0) into the values of P_i
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n_loc) return;
    constexpr int RF = thm_mesh::RF;
    if (dim == 2) {
        double g = 0, s = 0;
        for (int u = 0; u < RF; ++u) {
            const int32_t f = row_face[r * RF + u];
            if (f < 0) continue;
            const int a = row_face_a[r * RF + u];
            const double v = kwf[f] * face_mass(2, ref, X, face_v + (int64_t)f * 4, a, a);
            if (face_kind[f] == 1) g += v; else s += v;
        }
        bg64[r] = g; bs64[r] = tim * s; bg32[r] = (float)g; bs32[r] = (float)(tim * s);
        if (tre != 0.0 && s != 0.0) {
            const int64_t sl = r / SELL_C;
            const int lane = (int)(r % SELL_C);
            const int64_t base = slice_ptr[sl];
            const int w = (int)((slice_ptr[sl + 1] - base) / SELL_C);
            for (int t = 0; t < w; ++t) {
                const int64_t idx = base + (int64_t)t * SELL_C + lane;
                if (!pad[idx] && col[idx] == r) {
                    val64[idx] += tre * s;
                    val32[idx] = (float)val64[idx];
                }
            }
        }
        return;
    }
    bg64[r] = 0; bs64[r] = 0; bg32[r] = 0; bs32[r] = 0;
    const int64_t sl = r / SELL_C;
    const int lane = (int)(r % SELL_C);
    const int64_t base = slice_ptr[sl];
    const int w = (int)((slice_ptr[sl + 1] - base) / SELL_C);
    for (int t = 0; t < w; ++t) {
        const int64_t idx = base + (int64_t)t * SELL_C + lane;
        double g = 0, s = 0;
        if (!pad[idx]) {
            const int32_t cc = col[idx];
            for (int u = 0; u < RF; ++u) {
                const int32_t f = row_face[r * RF + u];
                if (f < 0) continue;
                const int a = row_face_a[r * RF + u], side = row_face_side[r * RF + u];
                for (int b = 0; b < fd; ++b) {
                    if (face_loc[((int64_t)f * 2 + side) * fd + b] != cc) continue;
                    const double v = kwf[f] * face_sgn[(int64_t)f * fd + a] * face_sgn[(int64_t)f * fd + b] *
                                     face_mass(3, ref, X, face_v + (int64_t)f * 4, a, b);
                    if (face_kind[f] == 1) g += v; else s += v;
                }
            }
        }
        bvg64[idx] = g; bvs64[idx] = tim * s; bvg32[idx] = (float)g; bvs32[idx] = (float)(tim * s);
        if (tre != 0.0 && s != 0.0) {
            val64[idx] += tre * s;
            val32[idx] = (float)val64[idx];
        }
    }
}

// Values of the interface-entry terms: kappa*omega times the signed face mass
// between DOFs a and b.
__global__ void k_iface_vals(int dim, int64_t n_terms, int fd, const double* __restrict__ ref,
                             const double* __restrict__ X, const int32_t* __restrict__ face_v,
                             const int8_t* __restrict__ face_sgn, const int32_t* __restrict__ tf,
                             const int8_t* __restrict__ ta, const int8_t* __restrict__ tb,
                             const double* __restrict__ kwf, double* __restrict__ val) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n_terms) return;
    const int32_t f = tf[p];
    const int a = ta[p], b = tb[p];
    val[p] = kwf[f] * face_sgn[(int64_t)f * fd + a] * face_sgn[(int64_t)f * fd + b] *
             face_mass(dim, ref, X, face_v + (int64_t)f * 4, a, b);
}

// Dirichlet values: tangential moments of E^inc(x) = pol exp(-i omega dir.x)
// along the global direction lo -> hi, by 8-point Gauss-Legendre on [0,1]:
//   Whitney DOF  m0 = l int_0^1 E_t(s) ds,
//   gradient DOF m1 = 3 l int_0^1 E_t(s) (1 - 2s) ds.
__constant__ double c_gl8_x[8] = {-0.9602898564975363, -0.7966664774136267, -0.5255324099163290,
                                  -0.1834346424956498, 0.1834346424956498,  0.5255324099163290,
                                  0.7966664774136267,  0.9602898564975363};
__constant__ double c_gl8_w[8] = {0.1012285362903763, 0.2223810344533745, 0.3137066458778873,
                                  0.3626837833783620, 0.3626837833783620, 0.3137066458778873,
                                  0.2223810344533745, 0.1012285362903763};

__global__ void k_dirichlet(int64_t n_de, int dim, int order, const int64_t* __restrict__ edges,
                            const double* __restrict__ X, const int64_t* __restrict__ elo,
                            const int64_t* __restrict__ ehi, const double* __restrict__ om, double pr0, double pi0,
                            double pr1, double pi1, double pr2, double pi2, double d0, double d1,
                            double d2, double2* __restrict__ uD) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n_de) return;
    int64_t e = edges[t];
    double xl[3] = {0, 0, 0}, tv[3] = {0, 0, 0};
    for (int k = 0; k < dim; ++k) {
        xl[k] = X[elo[e] * dim + k];
        tv[k] = X[ehi[e] * dim + k] - xl[k];
    }
    double l = sqrt(tv[0] * tv[0] + tv[1] * tv[1] + tv[2] * tv[2]);
    // pol . t_hat
    double ptr = (pr0 * tv[0] + pr1 * tv[1] + pr2 * tv[2]) / l;
    double pti = (pi0 * tv[0] + pi1 * tv[1] + pi2 * tv[2]) / l;
    const double omega = om[t];
    double m0r = 0, m0i = 0, m1r = 0, m1i = 0;
    for (int q = 0; q < 8; ++q) {
        double s = 0.5 * (c_gl8_x[q] + 1.0), wq = 0.5 * c_gl8_w[q];
        double ph = -omega * (d0 * (xl[0] + s * tv[0]) + d1 * (xl[1] + s * tv[1]) + d2 * (xl[2] + s * tv[2]));
        double sn, cs;
        sincos(ph, &sn, &cs);
        double er = ptr * cs - pti * sn, ei = ptr * sn + pti * cs;
        m0r += wq * er; m0i += wq * ei;
        m1r += wq * er * (1.0 - 2.0 * s); m1i += wq * ei * (1.0 - 2.0 * s);
    }
    if (order == 1) {
        uD[e] = make_double2(l * m0r, l * m0i);
    } else {
        uD[2 * e] = make_double2(l * m0r, l * m0i);
        uD[2 * e + 1] = make_double2(3.0 * l * m1r, 3.0 * l * m1i);
    }
}

// Dirichlet values given by the caller: u_D[ids[t]] = vals[t].
__global__ void k_dirichlet_given(int64_t n_dir, const int64_t* __restrict__ ids, const double2* __restrict__ vals,
                                  double2* __restrict__ uD) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < n_dir) uD[ids[t]] = vals[t];
}

// Lifting: f_i = -(P_i)_{F,D} u_D from the cells of each row (2-D: the face
// terms never couple a free DOF to a Dirichlet one).
__global__ void k_lifting(int dim, int64_t n_loc, int nb, int maxc, const double* __restrict__ ref,
                          const double* __restrict__ X, const int32_t* __restrict__ cells,
                          const int8_t* __restrict__ signs, const int32_t* __restrict__ cell_loc,
                          const int32_t* __restrict__ cell_dofs, const double* __restrict__ mu,
                          const double* __restrict__ w2c,
                          const int32_t* __restrict__ row_cell, const int32_t* __restrict__ row_k,
                          const double2* __restrict__ uD, int fd, const int32_t* __restrict__ face_v,
                          const int32_t* __restrict__ face_dof, const int8_t* __restrict__ face_sgn,
                          const int32_t* __restrict__ face_loc, const int32_t* __restrict__ row_face,
                          const int8_t* __restrict__ row_face_a, const int8_t* __restrict__ row_face_side,
                          const int8_t* __restrict__ face_kind, const double* __restrict__ kwf, double tre,
                          double tim, double2* __restrict__ f,
                          double2* __restrict__ fres) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n_loc) return;
    double fr = 0, fi = 0;
    for (int u = 0; u < maxc; ++u) {
        int32_t c = row_cell[r * maxc + u];
        if (c < 0) break;
        int kr = row_k[r * maxc + u];
        double hh[3];
        cell_sides(X, dim, cells, c, hh);
        for (int kc = 0; kc < nb; ++kc) {
            if (cell_loc[(int64_t)c * nb + kc] >= 0) continue;
            double s = (double)(signs[(int64_t)c * nb + kr] * signs[(int64_t)c * nb + kc]);
            double v = s * cell_entry(dim, ref, nb, mu[c], w2c[c], hh, kr, kc);
            double2 d = uD[cell_dofs[(int64_t)c * nb + kc]];
            fr -= v * d.x;
            fi -= v * d.y;
        }
    }
    // face terms coupling the row to Dirichlet DOFs: -(i kappa omega M_f) u_D.
    // The global system holds only the Gamma^inf faces; the subdomain operator
    // T_i also the transmission faces of Sigma, with the coefficient
    // (tre + i tim) kappa omega (3-D only: in 2-D no Dirichlet DOF lies on an
    // interface edge).
    double gr = fr, gi = fi;
    constexpr int RF = thm_mesh::RF;
    for (int u = 0; u < RF; ++u) {
        const int32_t f = row_face[r * RF + u];
        if (f < 0) continue;
        const int a = row_face_a[r * RF + u], side = row_face_side[r * RF + u];
        for (int b = 0; b < fd; ++b) {
            if (face_loc[((int64_t)f * 2 + side) * fd + b] >= 0) continue;
            const int32_t gd = face_dof[(int64_t)f * fd + b];
            const double v = kwf[f] * face_sgn[(int64_t)f * fd + a] * face_sgn[(int64_t)f * fd + b] *
                             face_mass(dim, ref, X, face_v + (int64_t)f * 4, a, b);
            const double2 d = uD[gd];
            if (face_kind[f] == 1) {
                fr += v * d.y;            // -(i v)(d.x + i d.y) = v d.y - i v d.x
                fi -= v * d.x;
                gr += v * d.y;
                gi -= v * d.x;
            } else {                      // -((tre + i tim) v) d
                fr -= v * (tre * d.x - tim * d.y);
                fi -= v * (tre * d.y + tim * d.x);
            }
        }
    }
    f[r] = make_double2(fr, fi);
    fres[r] = make_double2(gr, gi);
}

// ---------------------------------------------------------------------------
void assemble(thm_sys* s) {
    const thm_mesh* m = s->m;
    cudaStream_t st = s->st;
    const int nb = m->dpc;
    // omega per cell, face and Dirichlet edge (one value unless the mesh holds
    // a batch of independent problems)
    {
        auto prob = [&](int32_t sub) { return (sub < 0 || m->sub_prob.empty()) ? 0 : m->sub_prob[sub]; };
        THM_REQUIRE((int)s->omega_prob.size() == m->n_prob, "one omega per problem required");
        std::vector<double> w2h(m->n_cell), kwh(std::max<int64_t>(1, m->n_face), 0.0);
        std::vector<double> omh(std::max<size_t>(1, m->dir_edges.size()), 0.0);
        std::vector<double> eps;
        if (s->eps.p) s->eps.download(eps, st);
        for (int64_t c = 0; c < m->n_cell; ++c) {
            const double om = s->omega_prob[prob(m->cell_sub[c])];
            w2h[c] = om * om * (eps.empty() ? 1.0 : eps[c]);      // the mass term omega^2 eps_c M_c
        }
        for (int64_t f = 0; f < m->n_face; ++f) {
            const int32_t sb = m->face_sub[2 * f] >= 0 ? m->face_sub[2 * f] : m->face_sub[2 * f + 1];
            kwh[f] = s->kappa * s->omega_prob[prob(sb)];
        }
        if (!m->dir_edges.empty()) {
            const int nv = m->dim == 2 ? 4 : 8;
            std::vector<int32_t> vprob(m->n_vert, 0);
            for (int64_t c = 0; c < m->n_cell; ++c)
                for (int v = 0; v < nv; ++v) vprob[m->cells[c * nv + v]] = prob(m->cell_sub[c]);
            for (size_t t = 0; t < m->dir_edges.size(); ++t)
                omh[t] = s->omega_prob[vprob[m->edge_lo[m->dir_edges[t]]]];
        }
        s->w2c.upload(w2h, st);
        s->kwf.upload(kwh, st);
        s->omd.upload(omh, st);
    }
    s->dev_err.alloc(1);
    s->dev_err.zero(st);
    s->ref.alloc(8 * 144);
    s->ref.zero(st);
    THM_LAUNCH(THM_K_SETUP, st, k_ref_matrices<<<1, 256, 0, st>>>(m->dim, m->order, nb, s->ref.p));
    THM_CUDA(cudaGetLastError());
    s->val64.alloc(m->n_slots);
    s->val32.alloc(m->n_slots);
    const int th = 256;
    auto grid = [&](int64_t n) { return (unsigned)((n + th - 1) / th); };
    THM_LAUNCH(THM_K_SETUP, st, k_assemble<<<grid(m->n_loc), th, 0, st>>>(m->dim, m->n_loc, nb, m->maxc, s->ref.p, m->d_coords.p, m->d_cells.p,
                                              m->d_cell_signs.p, m->d_cell_loc.p, s->mu_inv.p, s->w2c.p,
                                              m->d_slice_ptr.p, m->d_sell_col.p, m->d_sell_pad.p,
                                              m->d_row_cell.p, m->d_row_k.p, s->val64.p, s->val32.p));
    THM_CUDA(cudaGetLastError());
    if (s->trans_re != 0.0) {
        // K_i^loc (no Sigma terms) keeps the values before the real Sigma part is added
        s->valK64.alloc(m->n_slots);
        s->valK32.alloc(m->n_slots);
        THM_CUDA(cudaMemcpyAsync(s->valK64.p, s->val64.p, m->n_slots * sizeof(double), cudaMemcpyDeviceToDevice, st));
        THM_CUDA(cudaMemcpyAsync(s->valK32.p, s->val32.p, m->n_slots * sizeof(float), cudaMemcpyDeviceToDevice, st));
    }
    s->bg64.alloc(m->n_loc); s->bs64.alloc(m->n_loc);
    s->bg32.alloc(m->n_loc); s->bs32.alloc(m->n_loc);
    const bool sellb = m->dim == 3;
    s->bvg64.alloc(sellb ? m->n_slots : 1); s->bvs64.alloc(sellb ? m->n_slots : 1);
    s->bvg32.alloc(sellb ? m->n_slots : 1); s->bvs32.alloc(sellb ? m->n_slots : 1);
    THM_LAUNCH(THM_K_SETUP, st, k_face_terms<<<grid(m->n_loc), th, 0, st>>>(
        m->dim, m->n_loc, m->fd, s->ref.p, m->d_coords.p, m->d_face_v.p, m->d_face_sgn.p, m->d_face_kind.p,
        m->d_face_loc.p, m->d_row_face.p, m->d_row_face_a.p, m->d_row_face_side.p, m->d_slice_ptr.p,
        m->d_sell_col.p, m->d_sell_pad.p, s->kwf.p, s->trans_re, s->trans_im, s->val64.p, s->val32.p, s->bg64.p,
        s->bs64.p, s->bg32.p, s->bs32.p, s->bvg64.p, s->bvs64.p, s->bvg32.p, s->bvs32.p));
    THM_CUDA(cudaGetLastError());
    const int64_t nterm = (int64_t)m->if_tf.size();
    s->if_val.alloc(nterm > 0 ? nterm : 1);
    if (nterm > 0) {
        THM_LAUNCH(THM_K_SETUP, st, k_iface_vals<<<grid(nterm), th, 0, st>>>(m->dim, nterm, m->fd, s->ref.p, m->d_coords.p,
                                                                            m->d_face_v.p, m->d_face_sgn.p, m->d_if_tf.p,
                                                                            m->d_if_ta.p, m->d_if_tb.p, s->kwf.p,
                                                                            s->if_val.p));
        THM_CUDA(cudaGetLastError());
    }
    s->uD.alloc(m->n_dof);
    s->uD.zero(st);
    if (s->dir_user) {
        const int64_t nd = (int64_t)m->dir_dofs.size();
        if (nd > 0) {
            THM_LAUNCH(THM_K_SETUP, st, k_dirichlet_given<<<grid(nd), th, 0, st>>>(nd, m->d_dir_dofs.p, s->dir_vals.p,
                                                                                  s->uD.p));
            THM_CUDA(cudaGetLastError());
        }
    } else if (!m->dir_edges.empty()) {
        THM_LAUNCH(THM_K_SETUP, st, k_dirichlet<<<grid((int64_t)m->dir_edges.size()), th, 0, st>>>(
            (int64_t)m->dir_edges.size(), m->dim, m->order, m->d_dir_edges.p, m->d_coords.p, m->d_edge_lo.p,
            m->d_edge_hi.p, s->omd.p, s->pol[0], s->pol[1], s->pol[2], s->pol[3], s->pol[4], s->pol[5],
            s->dir[0], s->dir[1], s->dir[2], s->uD.p));
        THM_CUDA(cudaGetLastError());
    }
    s->f_loc.alloc(m->n_loc);
    s->f_res.alloc(m->n_loc);
    THM_LAUNCH(THM_K_SETUP, st, k_lifting<<<grid(m->n_loc), th, 0, st>>>(
        m->dim, m->n_loc, nb, m->maxc, s->ref.p, m->d_coords.p, m->d_cells.p, m->d_cell_signs.p, m->d_cell_loc.p,
        m->d_cell_dofs.p, s->mu_inv.p, s->w2c.p, m->d_row_cell.p, m->d_row_k.p, s->uD.p, m->fd, m->d_face_v.p,
        m->d_face_dof.p, m->d_face_sgn.p, m->d_face_loc.p, m->d_row_face.p, m->d_row_face_a.p, m->d_row_face_side.p,
        m->d_face_kind.p, s->kwf.p, s->trans_re, s->trans_im, s->f_loc.p, s->f_res.p));
    THM_CUDA(cudaGetLastError());
    THM_CUDA(cudaStreamSynchronize(st));
}

}  // namespace thm
