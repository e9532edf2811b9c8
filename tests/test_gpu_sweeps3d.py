"""The band sweeps of the larger 3D levels, one launch a sweep, against the same
phases as one grid with software barriers: the same sums in the same order, so
bitwise equal solutions, residuals and single relaxations.  Levels on both sides
of the rule's line (4,000 ghosts FP64, 6,000 FP32), with and without a junction
zone, an even, an odd and the smallest number of sweeps that take the path, and
one below it."""
import numpy as np
import pytest

from paper_1111_0983_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n,nc,kw", [
    (1, 97, 25, {}), (0, 97, 25, {}), (0, 65, 17, {}), (1, 85, 22, dict(junction_sweeps=0)),
    (1, 129, 17, dict(lam=2)), (0, 85, 22, dict(lam=3, junction_sweeps=0)), (1, 97, 25, dict(lam=1)),
    (1, 161, 21, {}),
])
def test_sweep_launches_equal_one_grid(precision, n, nc, kw):
    from paper_1111_0983_gb300 import gcmg
    P = inputs.torus()
    S = gcmg.Solver(P.phi_grid(n), nc, precision=precision, rtol=1e-30, max_cycles=3, **kw)
    for l in range(S.nlev):
        S.set_bc_types(l, P.bc_types(S.ghosts(l)["B"]))
    G = S.ghosts(0)
    g = torch.from_numpy(P.g_values(G["B"], G["nu"], P.bc_types(G["B"]))).cuda()
    f = torch.from_numpy(P.f_grid(n)).cuda()
    S.set_rhs(f, g)
    start = torch.from_numpy(np.random.default_rng(n).standard_normal((n,) * 3)).cuda()
    start *= torch.from_numpy(S.node_types(0) & 3 > 0).cuda()
    runs = []
    for mode in (0, 2, 0):
        S.set_boundary3d(mode)
        u, r = torch.zeros_like(start), start.clone()
        rel = S.solve(u)["rel"]   # the tolerance is never reached: u holds the last cycle's
        S.relax(0, r, f, g)
        runs.append((u, rel, r))
    for u, rel, r in runs[1:]:
        assert torch.equal(u, runs[0][0])
        assert torch.equal(r, runs[0][2])
        np.testing.assert_array_equal(rel, runs[0][1])


@pytest.mark.parametrize("precision,n,nc", [(0, 65, 17), (1, 65, 17), (0, 129, 17), (1, 129, 17)])
def test_flat_domain_with_many_junctions(precision, n, nc):
    """The same on a flat ellipsoid with a hole whose boundary changes type along
    twelve curves (six sectors, another pattern below): the cluster programs on the
    coarser levels, the band sweeps and the zone alone on the finer ones."""
    from paper_1111_0983_gb300 import gcmg
    x = np.linspace(-1.0, 1.0, n)
    X, Y, Z = np.meshgrid(x, x, x, indexing="ij")
    body = np.sqrt((X / 0.85) ** 2 + (Y / 0.7) ** 2 + (Z / 0.42) ** 2) - 1.0
    phi = np.maximum(0.42 * body, 0.2 - np.sqrt((X - 0.1) ** 2 + (Y - 0.05) ** 2))
    S = gcmg.Solver(phi, nc, precision=precision, rtol=1e-30, max_cycles=3)
    for l in range(S.nlev):
        B = S.ghosts(l)["B"]
        S.set_bc_types(l, (np.sin(3 * np.arctan2(B[:, 1], B[:, 0]) + (B[:, 2] > 0)) > 0).astype(np.uint8))
    rng = np.random.default_rng(n)
    start = torch.from_numpy(rng.standard_normal((n,) * 3)).cuda()
    start *= torch.from_numpy(S.node_types(0) & 3 > 0).cuda()
    f = torch.from_numpy(rng.standard_normal((n,) * 3)).cuda()
    g = torch.from_numpy(rng.standard_normal(S.num_ghosts(0))).cuda()
    S.set_rhs(f, g)
    runs = []
    for mode in (0, 2):
        S.set_boundary3d(mode)
        u, r = torch.zeros_like(start), start.clone()
        rel = S.solve(u)["rel"]
        S.relax(0, r, f, g)
        runs.append((u, rel, r))
    assert torch.equal(runs[0][0], runs[1][0]) and torch.equal(runs[0][2], runs[1][2])
    np.testing.assert_array_equal(runs[0][1], runs[1][1])
