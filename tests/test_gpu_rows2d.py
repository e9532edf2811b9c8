"""The 2D passes over row segments (defects, descent, interpolation, correction
update) where a row's run of inside nodes ends at, just before and just past a
64-node segment: solves on superellipses whose middle rows hold 63, 64, 65 and
129 inside nodes, both forms, against the oracle's converged solution (1e-10,
the solves' bound in test_gpu_parity.py)."""
import numpy as np
import pytest

import oracle
from helpers import rel_maxdiff
from paper_1111_0983_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,run", [(129, 63), (129, 64), (129, 65), (257, 129)])
@pytest.mark.parametrize("precision", [0, 1])
def test_segment_edges(n, run, precision):
    from paper_1111_0983_gb300 import gcmg
    h = 2.0 / (n - 1)
    c = 0.5 * h if run % 2 == 0 else 0.0     # an even run is centred between two nodes
    r = (run / 2 - 0.25) * h
    x, y = inputs.coords(2, n)
    phi = np.ascontiguousarray(((x - c) ** 8 + (y - c) ** 8) ** 0.125 - r)
    assert (phi < 0).sum(1).max() == run
    f = np.cos(3 * x) * np.exp(y)
    O = oracle.Oracle(phi, 33)
    S = gcmg.Solver(phi, 33, precision=precision, rtol=1e-11)
    for l in range(S.nlev):
        types = (S.ghosts(l)["B"][:, 0] > 0.1).astype(np.uint8)
        S.set_bc_types(l, types)
        O.set_bc(l, types)
    G = S.ghosts(0)
    g = np.ascontiguousarray(np.sin(2 * G["B"][:, 0]) + G["B"][:, 1])
    S.set_rhs(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda())
    u = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    assert S.solve(u)["converged"]
    O.set_rhs(f, g)
    uo, _, ok = O.solve(rtol=1e-13, max_cycles=100)
    assert rel_maxdiff(u.cpu().numpy(), uo, O.types(0) > 0) <= 1e-10
