"""The defect of a solve (inside nodes and ghosts in one launch) against the one
of the residual entry point (a launch each, over the whole box): the same
expressions, so equal norms, from a random start whose largest defect lies at
the first, a middle or the last ghost, and after a cycle."""
import numpy as np
import pytest

from paper_1111_0983_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("domain,n,nc", [("disk", 33, 17), ("disk", 129, 17), ("flower", 257, 33), ("torus", 33, 17),
                                         ("torus", 97, 25)])
def test_solve_defect_equals_residual(domain, n, nc, precision):
    from paper_1111_0983_gb300 import gcmg
    P = getattr(inputs, domain)()
    S = gcmg.Solver(P.phi_grid(n), nc, precision=precision, rtol=1e-30, max_cycles=1)
    for l in range(S.nlev):
        S.set_bc_types(l, P.bc_types(S.ghosts(l)["B"]))
    G = S.ghosts(0)
    g = P.g_values(G["B"], G["nu"], P.bc_types(G["B"]))
    f = torch.from_numpy(P.f_grid(n)).cuda()
    u0 = torch.from_numpy(np.random.default_rng(n).standard_normal((n,) * P.dim)).cuda()
    u0 *= torch.from_numpy(S.node_types(0) & 3 > 0).cuda()
    for q in (0, len(g) // 2, len(g) - 1):
        gq = g.copy()
        gq[q] = 1e12
        S.set_rhs(f, torch.from_numpy(gq).cuda())
        u = u0.clone()
        r = torch.empty_like(u)
        first = S.residual(u, r)
        rel = S.solve(u)["rel"]
        np.testing.assert_allclose([rel[0], rel[-1]], [first, S.residual(u, r)], rtol=1e-15)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("domain,n,nc", [("disk", 33, 17), ("flower", 257, 33), ("torus", 97, 25)])
def test_largest_defect_at_inside_nodes(domain, n, nc, precision):
    """The same with the largest defect at an inside node (f = 1e12 there): the first
    and last of all, the ends of a row segment of 64 and of the next one, the shortest
    run's, and some drawn ones."""
    from paper_1111_0983_gb300 import gcmg
    P = getattr(inputs, domain)()
    S = gcmg.Solver(P.phi_grid(n), nc, precision=precision, rtol=1e-30, max_cycles=1)
    for l in range(S.nlev):
        S.set_bc_types(l, P.bc_types(S.ghosts(l)["B"]))
    G = S.ghosts(0)
    g = torch.from_numpy(P.g_values(G["B"], G["nu"], P.bc_types(G["B"]))).cuda()
    types = S.node_types(0) & 3
    inside = np.flatnonzero(types == 1)
    first = inside[np.r_[True, np.diff(inside) > 1]]
    last = inside[np.r_[np.diff(inside) > 1, True]]
    length = last - first + 1
    nodes = {inside[0], inside[-1], first[np.argmin(length)], *np.random.default_rng(n).choice(inside, 3)}
    longest = np.argmax(length)
    nodes |= {first[longest], last[longest]} | {first[longest] + k for k in (63, 64) if length[longest] > k}
    f0 = torch.from_numpy(P.f_grid(n)).cuda()
    u0 = torch.from_numpy(np.random.default_rng(n).standard_normal((n,) * P.dim)).cuda()
    u0 *= torch.from_numpy(types > 0).cuda()
    for p in nodes:
        f = f0.clone()
        f.view(-1)[int(p)] = 1e12
        S.set_rhs(f, g)
        u = u0.clone()
        r = torch.empty_like(u)
        before = S.residual(u, r)
        assert int(r.abs().argmax()) == p
        rel = S.solve(u)["rel"]
        np.testing.assert_allclose([rel[0], rel[-1]], [before, S.residual(u, r)], rtol=1e-15)
