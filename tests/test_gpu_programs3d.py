"""3D launch programs are built once: band-sweep blocks at creation, a level's
cluster program when its boundary types are set, or before the first solve where
they never are; none for the coarsest level, for a junction zone that is never
swept or in another launch mode.  Solutions as with one grid (launch mode 2), bit
by bit, before and after a change of the types."""
import pytest

from paper_1111_0983_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw,at_creation,with_types,after_change", [
    (dict(precision=1), 1, 2, 1), (dict(precision=0), 1, 2, 1), (dict(precision=1, junction_sweeps=0), 1, 1, 0),
    (dict(precision=1, lam=1), 0, 2, 1)])
def test_programs_are_built_once(kw, at_creation, with_types, after_change):
    """97^3, 49^3 and 25^3: band-sweep blocks and the zone alone on 97^3, band and zone
    on 49^3."""
    from paper_1111_0983_gb300 import gcmg
    P, n = inputs.torus(), 97
    built = [gcmg.program_build_counter()]

    def step():
        now = gcmg.program_build_counter()
        d, built[0] = now - built[0], now
        return d

    S = gcmg.Solver(P.phi_grid(n), 25, rtol=1e-30, max_cycles=2, **kw)
    assert [S.level_n(l) for l in range(S.nlev)] == [97, 49, 25]
    assert step() == at_creation
    types = []
    for l in range(S.nlev):
        types.append(P.bc_types(S.ghosts(l)["B"]))
        S.set_bc_types(l, types[l])
    G = S.ghosts(0)
    f = torch.from_numpy(P.f_grid(n)).cuda()
    S.set_rhs(f, torch.from_numpy(P.g_values(G["B"], G["nu"], types[0])).cuda())

    def solve():
        u = torch.zeros((n,) * 3, dtype=torch.float64, device="cuda")
        S.solve(u)
        return u

    assert step() == with_types
    u = solve()
    assert torch.equal(solve(), u)
    assert step() == 0
    S.set_bc_types(0, 1 - types[0])
    assert step() == after_change
    v = solve()
    assert step() == 0
    S.set_boundary3d(2)
    assert torch.equal(solve(), v)
    S.set_bc_types(0, types[0])
    assert torch.equal(solve(), u)
    assert step() == 0   # that mode takes none


def test_types_never_set():
    """All Dirichlet, as created: built by the first solve."""
    from paper_1111_0983_gb300 import gcmg
    P, n = inputs.torus(), 65
    S = gcmg.Solver(P.phi_grid(n), 17, precision=1, rtol=1e-30, max_cycles=2)
    built = gcmg.program_build_counter()
    f = torch.from_numpy(P.f_grid(n)).cuda()
    S.set_rhs(f, torch.ones(S.num_ghosts(0), dtype=torch.float64, device="cuda"))
    runs = []
    for mode in (0, 0, 2):
        S.set_boundary3d(mode)
        runs.append(torch.zeros((n,) * 3, dtype=torch.float64, device="cuda"))
        S.solve(runs[-1])
    assert gcmg.program_build_counter() - built == S.nlev - 1
    assert torch.equal(runs[0], runs[1]) and torch.equal(runs[0], runs[2])
