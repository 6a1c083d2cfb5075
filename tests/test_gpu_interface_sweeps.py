"""The interface GMRES runs no sweep beyond its last step: without relaxation (one
cycle at this tolerance) a solve takes one sweep for the right-hand side, one
per interface step, one for the residual at the end of the cycle and one with
the solution; and the counts of two solves agree to the last subdomain step,
since nothing is run on vectors that were not written."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mode", ["fp64", "mixed"])
@pytest.mark.parametrize("relax", [0, 1])
def test_sweeps_per_interface_step(mode, relax):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2105_11993_gb300 as thm
    P = W.square_problem(12, 2, 1, 9.0, mu_inv=W.mu_inv_lognormal(144, 0.3, "sweeps"))
    counts = []
    for _ in range(2):
        s = thm.System(thm.Mesh.from_workload(P.mesh, 1), P.mu_inv, 9.0, 1.0, P.pol, P.direction)
        _, st = s.solve(mode=mode, rtol=1e-6, max_refine=1, relax=relax, check=False)
        counts.append((st["sweeps"], st["inner_iters"], st["outer_iters"]))
        if not relax:
            assert st["sweeps"] == st["outer_iters"] + 3
    assert counts[0] == counts[1]


@pytest.mark.parametrize("mode", ["fp64", "mixed"])
def test_converged_problems_of_a_batch_take_no_steps(mode):
    """Three problems of different size end after different numbers of interface
    steps.  Those that have ended take no more subdomain steps while the others go
    on, whatever a solve before left in the workspace: a solve to a loose
    interface tolerance takes the same steps on a new system and after a solve to
    a tight one."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2105_11993_gb300 as thm
    ps = [W.square_problem(n, 2, 1, 9.0, mu_inv=W.mu_inv_lognormal(n * n, 0.3, "sweeps")) for n in (8, 12, 24)]
    mesh, _ = thm.Mesh.batch([p.mesh for p in ps], 1)
    mu = torch.cat([torch.tensor(p.mu_inv) for p in ps]).cuda()
    loose = dict(mode=mode, rtol=1e-2, outer_tol=1e-3, max_refine=1, check=False)
    counts = []
    for tight_before in (False, True):
        s = thm.System(mesh, mu, [9.0] * 3, 1.0, ps[0].pol, ps[0].direction)
        if tight_before:
            s.solve(mode=mode, rtol=1e-8, check=False)
        _, st = s.solve(**loose)
        counts.append((st["sweeps"], st["inner_iters"], st["outer_iters"]))
    assert counts[0] == counts[1]
