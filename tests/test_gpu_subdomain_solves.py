"""The subdomain solves of a sweep where their kernel takes another branch:
cycles that end at the restart length, FP32 cycles refined in FP64, complex
factors, few vectors per pass and many, subdomains whose columns need 32 bits
and whose Krylov vectors stay in global memory, against the oracle's sweep with
direct subdomain solves.

Tolerance: the solves stop at a residual of 1e-13 (or where a cycle no longer
halves it, about 1e-16 cond(T_i)), so x is within 1e-13 cond(T_i) of the
oracle's; cond(T_i) <= 1.5e4 for the small problems (computed), taken as 1e-8,
and about (order / (h omega))^2 * 1e2 = 1e6 for the large one, taken as 1e-6."""
import numpy as np
import pytest

import workloads as W
from oracle import ddm as odd
from test_gpu_parity import CASES as SMALL, make_system

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2105_11993_gb300 import build
    build.build()


def _long():
    """Two subdomains of more than 65,536 DOFs."""
    mesh = W.structured_mesh_2d(192, 92, 2, 1, bc="impedance", relabel=True, rotate_cells=True)
    pol, d = W.plane_wave_y(2)
    return W.Problem("long", mesh, 2, W.mu_inv_lognormal(mesh.n_cell, 0.1, "long"), 9.0, 1.0, pol, d)


PROBLEMS = dict(SMALL, long=_long)


@pytest.mark.parametrize("name,mode,precond,restart", [
    ("p2_rot", "fp64", "blockdiag", 8),        # restarted cycles (each falls by 0.25 or more)
    ("p2_rot", "mixed", "blockdiag", 8),
    ("p2_rot", "mixed", "full", 0),
    ("ragged_p2", "fp64", "full", 0),
    ("ragged_p2", "mixed", "blockdiag", 0),
    ("cube_ragged", "fp64", "blockdiag", 12),
    ("cube_ragged", "mixed", "blockdiag", 0),
    ("long", "fp64", "blockdiag", 0),
    ("long", "mixed", "blockdiag", 0),
])
def test_sweep_against_direct_subdomain_solves(name, mode, precond, restart):
    P = PROBLEMS[name]()
    mesh, s = make_system(P)
    D = odd.setup(P)
    recv, send, gdf = s.iface_dofs()
    okey = {}
    for p in D.pairs:
        for d in p.free:
            okey[(p.i, p.j, int(d))] = len(okey)
    perm = np.array([okey[(int(a), int(b), int(c))] for a, b, c in zip(recv, send, gdf)])
    rng = np.random.default_rng(5)
    g = 1e-2 * (rng.standard_normal(s.n_iface) + 1j * rng.standard_normal(s.n_iface))
    g_or = np.zeros_like(g)
    g_or[perm] = g
    ref, _ = odd.sweep(D, g_or, odd.local_sources(D), True, odd.subdomain_solver(D, "direct"))
    out, x, st = s.sweep(torch.tensor(g, device="cuda"), mode=mode, precond=precond, inner_restart=restart, inner_tol=1e-13)
    tol = 1e-6 if name == "long" else 1e-8
    assert np.linalg.norm(out.cpu().numpy() - ref[perm]) <= tol * np.linalg.norm(ref)
    # the same bits again: every sum has a fixed order
    out2, x2, _ = s.sweep(torch.tensor(g, device="cuda"), mode=mode, precond=precond, inner_restart=restart, inner_tol=1e-13)
    assert torch.equal(x, x2) and torch.equal(out, out2)
