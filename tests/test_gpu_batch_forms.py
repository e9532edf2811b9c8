"""Batched solves in every form of the relaxation launch -- one and two records
a thread, 512 threads (many extra sweeps: halos that cover the domain) -- with
the exact junction solve and with junction sweeps: every domain equals the
single-domain solver's solution to 1e-10 (the bound of test_gpu_batch.py)."""
import numpy as np
import pytest

from helpers import rel_maxdiff
from paper_1111_0983_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(), dict(lam=30), dict(lam=7, delta_over_h=6.0),
                                dict(junction_solve=0, junction_sweeps=3, junction_radius=2.0)])
def test_batch_equals_single(kw):
    from paper_1111_0983_gb300 import gcmg
    probs = [inputs.star(i, params=dict(inputs.star_params(i), n=n)) for i, n in ((0, 257), (1, 129), (5, 257))]
    sizes = [P.meta["n"] for P in probs]

    def data(S, P, n):
        for l in range(S.nlev):
            S.set_bc_types(l, P.bc_types(S.ghosts(l)["B"]))
        G = S.ghosts(0)
        g = P.g_values(G["B"], G["nu"], P.bc_types(G["B"]))
        S.set_rhs(torch.from_numpy(P.f_grid(n)).cuda(), torch.from_numpy(g).cuda())

    B = gcmg.Batch([P.phi_grid(n) for P, n in zip(probs, sizes)], 33, rtol=1e-11, max_cycles=200, **kw)
    for S, P, n in zip(B.domains, probs, sizes):
        data(S, P, n)
    for _ in range(2):   # the second solve finds the first one's grids
        stats, _ = B.solve()
    assert all(s["converged"] for s in stats)
    for k, (P, n) in enumerate(zip(probs, sizes)):
        S = gcmg.Solver(P.phi_grid(n), 33, precision=1, rtol=1e-11, max_cycles=200, **kw)
        data(S, P, n)
        u = torch.zeros((n, n), dtype=torch.float64, device="cuda")
        assert S.solve(u)["converged"]
        ub = torch.zeros_like(u)
        B.solution(k, ub)
        assert rel_maxdiff(ub.cpu().numpy(), u.cpu().numpy(), (S.node_types(0) & 3) > 0) <= 1e-10


@pytest.mark.parametrize("kw,more", [(dict(), 9), (dict(junction_solve=0, junction_sweeps=3, junction_radius=2.0), 6)])
def test_blocks_too_large_for_the_merged_launch(kw, more):
    """A band of 2 h with 60 sweeps at 513^2: blocks of more than 4,096 staged nodes,
    whose depth takes strips, blocks, their write-back and the junction zone as
    launches of their own (by the launch counter: three, with junction sweeps two,
    more for each of that depth's three relaxations)."""
    from paper_1111_0983_gb300 import gcmg
    probs = [inputs.star(i, params=dict(inputs.star_params(i), n=n)) for i, n in ((0, 513), (3, 257))]
    sizes = [P.meta["n"] for P in probs]

    def data(S, P, n):
        for l in range(S.nlev):
            S.set_bc_types(l, P.bc_types(S.ghosts(l)["B"]))
        G = S.ghosts(0)
        g = P.g_values(G["B"], G["nu"], P.bc_types(G["B"]))
        S.set_rhs(torch.from_numpy(P.f_grid(n)).cuda(), torch.from_numpy(g).cuda())

    def batch(lam):
        B = gcmg.Batch([P.phi_grid(n) for P, n in zip(probs, sizes)], 33, rtol=1e-11, max_cycles=200, lam=lam,
                       delta_over_h=2.0, **kw)
        for S, P, n in zip(B.domains, probs, sizes):
            data(S, P, n)
        B.solve()
        before = gcmg.launch_counter()   # the second solve finds the first one's grids
        stats, steps = B.solve()
        assert all(s["converged"] for s in stats)
        return B, (gcmg.launch_counter() - before - 2) // steps

    B, launches = batch(60)
    assert launches - batch(5)[1] == more
    for k, (P, n) in enumerate(zip(probs, sizes)):
        S = gcmg.Solver(P.phi_grid(n), 33, precision=1, rtol=1e-11, max_cycles=200, lam=60, delta_over_h=2.0, **kw)
        data(S, P, n)
        u = torch.zeros((n, n), dtype=torch.float64, device="cuda")
        assert S.solve(u)["converged"]
        ub = torch.zeros_like(u)
        B.solution(k, ub)
        assert rel_maxdiff(ub.cpu().numpy(), u.cpu().numpy(), (S.node_types(0) & 3) > 0) <= 1e-10
