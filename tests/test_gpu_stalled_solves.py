"""Bounded waits of the subdomain solves: with the table copies held back (test
switch, 20 ms limit) a sweep, a solve and an adjoint report THM_ETIMEOUT, and
the next call on the same system gives what it gave before: the same bits, since
every sum has a fixed order."""
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


@pytest.mark.parametrize("mode", ["fp64", "mixed"])
def test_stalled_calls_report_a_timeout(mode, monkeypatch):
    import paper_2105_11993_gb300 as thm
    P = W.square_problem(12, 2, 1, 9.0, mu_inv=W.mu_inv_lognormal(144, 0.3, "stall"))
    mesh = thm.Mesh.from_workload(P.mesh, P.order)
    s = thm.System(mesh, P.mu_inv, P.omega, P.kappa, P.pol, P.direction)
    g = 1e-2 * torch.randn(s.n_iface, dtype=torch.complex128, device="cuda",
                           generator=torch.Generator("cuda").manual_seed(1))
    u, _ = s.solve(mode=mode, rtol=1e-8)
    calls = {
        "sweep": lambda: s.sweep(g, mode=mode)[:2],
        # one interface step: every sweep of a stalled solve waits out its limit
        "solve": lambda: s.solve(mode=mode, rtol=1e-8, max_refine=1, outer_maxit=1, check=False)[:1],
        "adjoint": lambda: s.adjoint(u, u.conj(), mode=mode, rtol=1e-8)[:1],
    }
    monkeypatch.setenv("THM_BT_WAIT_LIMIT_MS", "20")
    for name, call in calls.items():
        before = call()
        monkeypatch.setenv("THM_TEST_STALL_TMA", "1")
        if name == "solve":
            assert s.solve(mode=mode, rtol=1e-8, max_refine=1, outer_maxit=1, check=False)[1]["status"] == -5
        else:
            with pytest.raises(thm.ThmError) as e:
                call()
            assert e.value.code == -5, name
        monkeypatch.delenv("THM_TEST_STALL_TMA")
        for a, b in zip(before, call()):
            assert torch.equal(a, b), name
