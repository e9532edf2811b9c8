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
