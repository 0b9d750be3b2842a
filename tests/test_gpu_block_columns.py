"""A column of a block of right-hand sides gets the arithmetic of a single column, bit for bit, also where the
interiors have several block rows per 256-wide diagonal block (their sweeps then go by whole diagonal blocks):
operators on 1 to 8 columns, two and three levels, and ragged last blocks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1201_5991_gb300 import meshgen
from paper_1201_5991_gb300.solver import BddcSolver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("prob", [lambda: meshgen.elasticity3d(16, 2, seed=4),             # interiors of 17 block rows
                                  lambda: meshgen.elasticity3d(16, 4, seed=4, group=2),    # level 2 of several
                                  lambda: meshgen.elasticity3d_tet(12, 8, seed=1)])        # uneven
def test_operators_on_blocks_match_single_columns(prec, prob):
    s = BddcSolver(prob(), precision=prec)
    R = torch.tensor(np.random.default_rng(3).standard_normal((8, s.n_iface)), dtype=torch.float64, device="cuda")
    ops = [s.apply_precond, s.apply_schur] + ([s.apply_inner_schur] if prec == "mixed" else [])
    for op in ops:
        one = torch.stack([op(R[k].contiguous()) for k in range(8)])
        for w in (2, 3, 4, 5, 8):
            assert torch.equal(op(R[:w].contiguous()), one[:w]), (op.__name__, w)
