"""The explicit inverse of the coarsest factor (mixed precision): only the blocks on and below the diagonal are
substituted, the rest is mirrored.

The preconditioner against the FP64 one, whose coarse solves are FP64 sweeps, on subdomains of two elements a side
so that the coarse problem dominates.  Bound 1e-2, the one tests/test_gpu_interface_inverse.py derives for the
FP32 local solves; a block that is not mirrored, or a column that starts at the wrong block, gives O(1).  Coarse sizes: less
than one tile (4 subdomains), a few tiles with a ragged last one, one past 2,048 (32 tiles and
more), and the signed factor of the Stokes cavity."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1201_5991_gb300 import meshgen
from paper_1201_5991_gb300.solver import BddcSolver

pytestmark = pytest.mark.gpu

CASES = {
    "one_tile": lambda: meshgen.elasticity3d(4, 2, seed=1),
    "few_tiles": lambda: meshgen.elasticity3d(6, 3, seed=2),
    "many_tiles": lambda: meshgen.elasticity3d(16, 8, seed=3),
    "corners": lambda: meshgen.poisson2d(24, 12),
    "cavity": lambda: meshgen.stokes_cavity(6, 3),
}


@pytest.mark.parametrize("name", list(CASES))
def test_coarse_inverse(name):
    p = CASES[name]()
    s64 = BddcSolver(p, precision="fp64")
    R = torch.tensor(np.random.default_rng(4).standard_normal((3, s64.n_iface)), dtype=torch.float64, device="cuda")
    ref = s64.apply_precond(R).cpu().numpy()
    got = BddcSolver(p, precision="mixed").apply_precond(R).cpu().numpy()
    err = max(np.linalg.norm(got[k] - ref[k]) / np.linalg.norm(ref[k]) for k in range(3))
    print(f"{name}: FP32 preconditioner error vs FP64 with the coarse inverse {err:.2e}")
    assert err < 1e-2
