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
