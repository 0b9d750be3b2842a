"""The store of search directions that a refined solve keeps for its later inner solves, where device memory
runs out: bddc_alloc_probe makes the allocation fail on the host.  The handle stays usable and other handles,
which allocate from the same pool, keep their data."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem
from paper_1201_5991_gb300 import capi, meshgen
from paper_1201_5991_gb300.solver import BddcSolver

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.fixture
def probe():
    yield capi.lib().bddc_alloc_probe
    capi.lib().bddc_alloc_probe(0)


def test_growth_that_fails_leaves_no_freed_memory_in_use(probe):
    p = meshgen.elasticity3d(8, 4, seed=4, nrhs=8)
    ref = fem.direct_solve(p)
    a = BddcSolver(p, precision="mixed")
    F = _dev(p.f.T)
    one = a.solve(F[0].contiguous(), tol=1e-10)          # the store of one column
    a.apply_schur(torch.zeros(8, a.n_iface, dtype=torch.float64, device="cuda"))   # every other buffer of a block
    again = a.solve(F[0].contiguous(), tol=1e-10)
    assert torch.equal(one, again)
    probe(a.last_stats.factor_bytes)                       # no room for the store of a block
    try:
        U = a.solve(F, tol=1e-10).cpu().numpy()
        assert all(_rel(U[k], ref[:, k]) < 1e-7 for k in range(8))
    except capi.BddcError as e:
        assert e.code == capi.ERR_OOM
    probe(0)
    b = BddcSolver(p, precision="mixed")                   # takes what the failed growth gave back
    r = _dev(np.random.default_rng(1).standard_normal(b.n_iface))
    z = b.apply_precond(r)
    for k in range(3):
        assert _rel(a.solve(F[k].contiguous(), tol=1e-10).cpu().numpy(), ref[:, k]) < 1e-7
    assert torch.equal(b.apply_precond(r), z)


def test_held_bytes_count_the_store_once():
    p = meshgen.elasticity3d(8, 4, seed=4, nrhs=8)
    F = _dev(p.f.T)
    held = []
    for first in (True, False):   # the store grows from one column to eight, or starts with eight
        s = BddcSolver(p, precision="mixed")
        if first:
            s.solve(F[0].contiguous(), tol=1e-10)
        s.solve(F, tol=1e-10)
        held.append(s.last_stats.factor_bytes)
    assert held[0] == held[1]


def test_first_solve_allocates_nothing(probe):
    p = meshgen.elasticity3d(8, 4, seed=4)
    ref = fem.direct_solve(p)[:, 0]
    for prec in ("mixed", "fp64"):
        s = BddcSolver(p, precision=prec)
        probe(1)                                           # no further allocation of a handle succeeds
        assert _rel(s.solve(_dev(p.f[:, 0]), tol=1e-10).cpu().numpy(), ref) < 1e-7
        probe(0)


def test_solves_with_less_store_or_none(probe):
    # a block's store takes 8 columns; the column's own 128 directions make room for 16 of each, one byte less for
    # 8 (fewer than the iterations of one solve), and less than a sixteenth of them for none
    p = meshgen.elasticity3d(8, 4, seed=4, nrhs=8)
    ref = fem.direct_solve(p)
    F = _dev(p.f.T)
    its = {}
    for room in ("all", "16", "8", "none"):
        s = BddcSolver(p, precision="mixed")
        s.apply_schur(torch.zeros(8, s.n_iface, dtype=torch.float64, device="cuda"))
        s.solve(F[0].contiguous(), tol=1e-10)
        held, store = s.last_stats.factor_bytes, 128 * 8 * s.n_iface
        probe({"all": 0, "16": held, "8": held - 1, "none": held - store * 31 // 32}[room])
        U = s.solve(F, tol=1e-10).cpu().numpy()
        assert s.last_stats.converged == 1
        its[room] = s.last_stats.iterations
        assert all(_rel(U[k], ref[:, k]) < 1e-7 for k in range(8)), room
        assert torch.equal(s.solve(F, tol=1e-10), s.solve(F, tol=1e-10)), room
        grown = s.last_stats.factor_bytes - held
        assert {"all": grown > 6 * store, "16": grown == 0, "8": -store < grown < 0, "none": grown <= -store}[room], room
        probe(0)
    assert its["all"] <= its["16"] <= its["none"] and its["8"] <= its["none"], its


def test_directions_are_forgotten_when_the_inner_operator_changes():
    # a tolerance below what FP64 reaches: the outer steps stagnate, the inner operator becomes the FP64 one, whose
    # solves start from its own directions; neither that solve nor the next, with the first operator again, is wrong
    p = meshgen.elasticity3d(8, 4, seed=4, nrhs=2)
    ref = fem.direct_solve(p)
    s = BddcSolver(p, precision="mixed")
    f = _dev(p.f[:, 0])
    before = s.solve(f, tol=1e-10)
    u = s.solve(f, tol=1e-18, allow_not_converged=True)
    assert s.last_stats.outer_iterations > 6 and s.last_stats.rel_residual < 1e-12
    assert _rel(u.cpu().numpy(), ref[:, 0]) < 1e-9
    assert torch.equal(s.solve(f, tol=1e-10), before)
    U = s.solve(_dev(p.f.T), tol=1e-18, allow_not_converged=True).cpu().numpy()
    assert all(_rel(U[k], ref[:, k]) < 1e-9 for k in range(2))
