"""The preconditioner's local solves with the explicit interface inverse (mixed precision, the inverse rows
go through the panel solves and updates of the factorisation) against the FP64 preconditioner.

Bound: the one tests/test_gpu_tc_panels.py has for the preconditioner of a tensor-core factor, 1e-2 (the
factor's 2^-22 products amplified by kappa(A_i) <= 1e4; the inverse adds products of the same relative error).
An inverse row that is dropped, shifted by a tile or started at the wrong panel gives O(1).  Cases:
interfaces of one tile (nGb = 1) and interiors smaller than a panel, interiors that end inside a 256-wide
sub-panel and inside a 512-wide super-panel (inner_operator = 1 keeps them unpadded, 2 pads them), subdomains
of unequal block counts, a last panel that holds no trailing factor column, and three levels; one column and
five (groups of 4 and 1 in the symmetric product; the same FP32 operations per column)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1201_5991_gb300 import meshgen
from paper_1201_5991_gb300.solver import BddcSolver

pytestmark = pytest.mark.gpu

CASES = {
    "poisson_8x8": lambda: meshgen.poisson2d(32, 4),                     # nI = 49: one tile each
    "poisson_32x32": lambda: meshgen.poisson2d(96, 3),                   # 16 interior tiles, two interface tiles
    "elast_5": lambda: meshgen.elasticity3d(10, 2, seed=9),              # interiors of 4 to 6 tiles
    "elast_8": lambda: meshgen.elasticity3d(16, 2, seed=3),              # interiors of 17 to 24 tiles
    "tet": lambda: meshgen.elasticity3d_tet(10, 9, seed=4),              # unequal block counts
    "kmeans_3lev": lambda: meshgen.elasticity3d_kmeans(12, 16, 4, seed=3, seed2=33),
}


@pytest.mark.parametrize("inner_operator", [1, 2])
@pytest.mark.parametrize("name", list(CASES))
def test_interface_inverse(name, inner_operator):
    p = CASES[name]()
    s64 = BddcSolver(p, precision="fp64")
    rng = np.random.default_rng(11)
    R = torch.tensor(rng.standard_normal((5, s64.n_iface)), dtype=torch.float64, device="cuda")
    ref = s64.apply_precond(R).cpu().numpy()
    s = BddcSolver(p, precision="mixed", inner_operator=inner_operator)
    one = s.apply_precond(R[0].contiguous()).cpu().numpy()
    blk = s.apply_precond(R).cpu().numpy()
    np.testing.assert_allclose(blk[0], one, rtol=0, atol=1e-5 * np.abs(one).max())
    err = max(np.linalg.norm(blk[k] - ref[k]) / np.linalg.norm(ref[k]) for k in range(5))
    print(f"{name}: FP32 preconditioner error vs FP64 with the interface inverse {err:.2e}")
    assert err < 1e-2
