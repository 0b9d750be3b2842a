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


def test_compact_operators_match():
    # interiors of 17 block rows: sweeps by 256-wide diagonal blocks against plain ones, and the interface inverse
    # against interface sweeps; S x is refined to FP64 accuracy (1e-11: kappa(K_II) 2^-53 and some), the preconditioner
    # has the tensor-core factor's accuracy (1e-2, as in test_gpu_tc_panels.py)
    p = meshgen.elasticity3d(16, 2, seed=4)
    full = BddcSolver(p, precision="mixed")
    full.solve(_dev(p.f[:, 0]), tol=1e-10)
    held, small = full.last_stats.factor_bytes, None
    try:
        for step in range(40):
            capi.lib().bddc_alloc_probe(int(held * (1.2 - 0.025 * step)))
            s = BddcSolver(p, precision="mixed")
            s.solve(_dev(p.f[:, 0]), tol=1e-10)
            if s.last_stats.factor_bytes < 0.9 * (held - 1024 * s.n_iface):
                small = s
                break
    finally:
        capi.lib().bddc_alloc_probe(0)
    assert small is not None
    R = _dev(np.random.default_rng(2).standard_normal((3, full.n_iface)))
    for op, tol in (("apply_schur", 1e-11), ("apply_precond", 1e-2)):
        a, b = getattr(full, op)(R), getattr(small, op)(R)
        assert float((a - b).norm() / a.norm()) < tol, op
