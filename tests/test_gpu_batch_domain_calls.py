"""A batch solves from the arrays its domains hold now: single calls on a domain
that move them (the first FP64 relaxation adds the FP64 inverses, the junction
blocks' switch rebuilds the junction programs) leave the batch's next solve
as it was, bit by bit."""
import numpy as np
import pytest

from paper_1111_0983_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(), dict(junction_solve=0, junction_sweeps=3, junction_radius=2.0)])
def test_batch_after_calls_on_a_domain(kw):
    from paper_1111_0983_gb300 import gcmg
    probs = [inputs.star(i) for i in (0, 1)]
    n = 129
    B = gcmg.Batch([P.phi_grid(n) for P in probs], 33, rtol=1e-10, **kw)
    data = []
    for S, P in zip(B.domains, probs):
        for l in range(S.nlev):
            S.set_bc_types(l, P.bc_types(S.ghosts(l)["B"]))
        G = S.ghosts(0)
        g = P.g_values(G["B"], G["nu"], P.bc_types(G["B"]))
        data.append((torch.from_numpy(P.f_grid(n)).cuda(), torch.from_numpy(g).cuda()))
        S.set_rhs(*data[-1])

    def solve():
        stats, _ = B.solve()
        us = [torch.zeros((n, n), dtype=torch.float64, device="cuda") for _ in probs]
        for k, u in enumerate(us):
            B.solution(k, u)
        return us, [s["rel"] for s in stats]

    us, rels = solve()
    for move in (lambda S: S.relax(0, us[0].clone(), *data[0]), lambda S: S.set_junction_blocks(True)):
        move(B.domains[0])
        # what the next allocations hold is neither an inverse nor a list
        junk = [torch.full((1 << 18,), float("nan"), device="cuda") for _ in range(4)]
        again, rels2 = solve()
        del junk
        for a, b in zip(us, again):
            assert torch.equal(a, b)
        for a, b in zip(rels, rels2):
            np.testing.assert_array_equal(a, b)


def test_batch_after_a_refused_solve():
    """A solve that is refused for one domain's junction zone (beyond 4,096 nodes a
    component) leaves the other's rebuilt on the host and not yet on the device; the
    autotuner then takes neither, and the next solve is that of a new batch."""
    from paper_1111_0983_gb300 import gcmg
    sizes = (257, 65)
    probs = [inputs.star(i, params=dict(inputs.star_params(i), n=n)) for i, n in zip((0, 1), sizes)]

    def batch():
        B = gcmg.Batch([P.phi_grid(n) for P, n in zip(probs, sizes)], 33, rtol=1e-10, junction_radius=64.0)
        for S, P, n in zip(B.domains, probs, sizes):
            G = S.ghosts(0)
            g = P.g_values(G["B"], G["nu"], np.zeros(len(G["B"]), np.uint8))
            S.set_rhs(torch.from_numpy(P.f_grid(n)).cuda(), torch.from_numpy(g).cuda())
        return B

    def mixed(S, on):   # types change across x = 0.05, or all Dirichlet
        for l in range(S.nlev):
            S.set_bc_types(l, ((S.ghosts(l)["B"][:, 0] > 0.05) & on).astype(np.uint8))

    def solve(B):
        B.solve()
        us = [torch.zeros((n, n), dtype=torch.float64, device="cuda") for n in sizes]
        for k, u in enumerate(us):
            B.solution(k, u)
        return us

    B = batch()
    mixed(B.domains[1], True)
    solve(B)
    mixed(B.domains[0], True)
    mixed(B.domains[1], False)
    with pytest.raises(gcmg.GcmgError, match="4096"):
        B.solve()
    B.autotune()
    B.set_tiles(0)
    mixed(B.domains[0], False)
    for a, b in zip(solve(B), solve(batch())):
        assert torch.equal(a, b)
