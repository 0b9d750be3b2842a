"""K_Ci where a level's largest constraint count exceeds 96: G is factored by panels of 16 columns on one SM per
subdomain and inverted over the whole chip (smaller levels take one block per subdomain, which
tests/test_gpu_coarse.py covers).  Same oracle and tolerance as there: FP64 form, 1e-10 relative Frobenius norm per
subdomain.  The subdomains' counts range from 27 to 192, so panels and warps of columns end ragged and the launch's
sizes exceed most subdomains'."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.bddc import Bddc
from paper_1201_5991_gb300 import meshgen
from paper_1201_5991_gb300.solver import BddcSolver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nsub", [(8, 20), (10, 24)])
def test_coarse_matrices_with_many_constraints(n, nsub):
    p = meshgen.elasticity3d_tet(n, nsub, seed=1)
    d = Bddc(p).levels[0]
    kc = BddcSolver(p, precision="fp64").coarse_matrices(1)
    assert max(k.shape[0] for k in kc) > 96 and len(kc) == len(d.KC)
    worst = max(np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in zip(kc, d.KC))
    print(f"tetrahedra {n}/{nsub}: FP64 K_Ci max relative error {worst:.2e}")
    assert worst < 1e-10
