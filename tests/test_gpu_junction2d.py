"""The 2D junction solve in one launch (FP32 cycles) at zones of a few nodes, of
the default size and of more equations than a CTA's threads hold at once, and on
domains without a junction: mixed solves against the oracle's converged
solution (1e-10), and the split relaxation against the merged one, bitwise."""
import numpy as np
import pytest

import oracle
from helpers import rel_maxdiff
from paper_1111_0983_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [1.0, 6.0, 20.0, 36.0])
@pytest.mark.parametrize("domain", ["flower", "star", "disk"])
def test_junction_zone_sizes(domain, radius):
    from paper_1111_0983_gb300 import gcmg
    P = {"flower": inputs.flower, "star": lambda: inputs.star(7), "disk": inputs.disk}[domain]()
    n, nc = 257, 33
    phi = P.phi_grid(n)
    O = oracle.Oracle(phi, nc, junction_radius=radius)
    S = gcmg.Solver(phi, nc, precision=1, rtol=1e-11, junction_radius=radius)
    for l in range(S.nlev):
        types = P.bc_types(S.ghosts(l)["B"])
        S.set_bc_types(l, types)
        O.set_bc(l, types)
    G = S.ghosts(0)
    f, g = P.f_grid(n), P.g_values(G["B"], G["nu"], P.bc_types(G["B"]))
    S.set_rhs(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda())
    O.set_rhs(f, g)
    uo, _, _ = O.solve(rtol=1e-13, max_cycles=200)
    runs = []
    for split in (0, 1):
        S.set_split2d(split)
        u = torch.zeros((n, n), dtype=torch.float64, device="cuda")
        assert S.solve(u)["converged"]
        runs.append(u)
    assert torch.equal(runs[0], runs[1])
    assert rel_maxdiff(runs[0].cpu().numpy(), uo, O.types(0) > 0) <= 1e-10
