"""Subdomains that fill the shared memory of one CTA: more of them than SMs (one
CTA each would do for the SMs), of sizes at which an apply or a default solve
does not fit one CTA, and a single one at the limit of eight CTAs.

T_i u = f holds for the u of a sweep with zero interface data to the tolerance
of the subdomain solves (1e-11, times the number of subdomains that end just
above it: 1e-10 of the whole); P_i P_i^{-1} x = x as in the tests of the
elimination tree (kappa = 0), to 1e-8."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2105_11993_gb300 import build
    build.build()


def _system(cells, s, order, kappa):
    import paper_2105_11993_gb300 as thm
    mesh = W.structured_mesh_2d(cells * s, cells * s, s, s)
    mu = W.mu_inv_lognormal(mesh.n_cell, 0.3, "large")
    pol, d = W.plane_wave_y(2)
    return thm, thm.System(thm.Mesh.from_workload(mesh, order), mu, 5.0, kappa, pol, d)


@pytest.mark.parametrize("cells,s,order", [(40, 13, 2), (39, 13, 2), (74, 13, 1), (77, 13, 1), (170, 1, 1)])
def test_sweep(cells, s, order):
    thm, sysg = _system(cells, s, order, 1.0)
    g = torch.zeros(max(1, sysg.n_iface), dtype=torch.complex128, device="cuda")
    f = sysg.local_sources()
    for mode in ("fp64", "mixed"):
        u = sysg.sweep(g, mode=mode)[1]
        r = sysg.apply_local(thm.OP_T, u, mode="fp64") - f
        assert float(r.norm() / f.norm()) <= 1e-10, mode


@pytest.mark.parametrize("cells,s,order", [(40, 13, 2), (77, 13, 1)])
def test_apply(cells, s, order):
    thm, sysg = _system(cells, s, order, 0.0)
    x = torch.randn(sysg.n_local, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(8))
    y = sysg.apply_local(thm.OP_PINV, x, mode="fp64")
    assert float((sysg.apply_local(thm.OP_T, y, mode="fp64") - x).norm() / x.norm()) <= 1e-8
