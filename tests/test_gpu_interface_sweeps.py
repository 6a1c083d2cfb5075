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
