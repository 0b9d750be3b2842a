"""Set-up where the interface inverses and the other memory that only saves time do not fit: it is made again in
the compact form, whose handles hold less and answer the same.  bddc_alloc_probe stands for a full device."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem
from paper_1201_5991_gb300 import capi, meshgen
from paper_1201_5991_gb300.solver import BddcSolver

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("prob", [lambda: meshgen.elasticity3d(12, 2, seed=4),
                                  lambda: meshgen.elasticity3d(12, 4, seed=4, group=2),   # three levels
                                  lambda: meshgen.stokes_cavity(8, 2)])
def test_setup_that_does_not_fit_is_made_compact(prob):
    p = prob()
    ref = fem.direct_solve(p)
    F = _dev(p.f.T)
    full = BddcSolver(p, precision="mixed")
    full.solve(F, tol=1e-12)
    held, smallest = full.last_stats.factor_bytes, None
    rest = held - 1024 * full.n_iface - 40000   # without the store of directions, which may shrink by itself
    try:
        for step in range(40):
            capi.lib().bddc_alloc_probe(int(held * (1.2 - 0.025 * step)))
            try:
                s = BddcSolver(p, precision="mixed")
            except capi.BddcError as e:
                assert e.code == capi.ERR_OOM
                break
            finally:
                capi.lib().bddc_alloc_probe(0)
            U = s.solve(F, tol=1e-12).cpu().numpy()
            smallest = s.last_stats.factor_bytes
            assert s.last_stats.converged == 1
            for k in range(U.shape[0]):
                assert np.linalg.norm(U[k] - ref[:, k]) < 1e-7 * np.linalg.norm(ref[:, k]), (step, k)
    finally:
        capi.lib().bddc_alloc_probe(0)
    assert smallest is not None and smallest < 0.9 * rest, (smallest, rest, held)


def test_forms_of_one_shape_are_tuned_apart():
    # a handle without the interface inverse has interface sweeps to tune, whatever was cached for one with it
    p = meshgen.poisson2d(91, 7)   # 49 subdomains: a shape of this test alone
    assert BddcSolver(p, precision="mixed").stats().tune_ms > 0
    assert BddcSolver(p, precision="mixed").stats().tune_ms == 0
    assert BddcSolver(p, precision="mixed", tensor_cores=2).stats().tune_ms > 0
