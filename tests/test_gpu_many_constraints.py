"""Subdomains with several hundred constraints, whose G is factored by panels in shared memory (more than its default
limit from 361 constraints on) and inverted over the whole chip: handles set up from several threads at once get what
each gets alone, and the mixed form's K_Ci keeps the FP32 factor's accuracy.  A ball of elements in the middle of
the cube is one subdomain with a hundred neighbours."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.bddc import Bddc
from paper_1201_5991_gb300 import meshgen
from paper_1201_5991_gb300.solver import BddcSolver

pytestmark = pytest.mark.gpu


def _ball(n, nsub, radius):
    p = meshgen.elasticity3d_tet(n, nsub, seed=1)
    c = p.coords[p.conn].mean(1)
    lo, hi = p.coords.min(0), p.coords.max(0)
    part = p.parts[0].copy()
    part[np.linalg.norm((c - lo) / (hi - lo) - 0.5, axis=1) < radius] = part.max() + 1
    u, part = np.unique(part, return_inverse=True)
    p.parts[0], p.n_parts[0] = part.astype(np.int32), len(u)
    return p


def test_setups_from_several_threads():
    probs = [_ball(12, 80, 0.3), _ball(14, 120, 0.3)]   # up to 543 and 615 constraints
    alone = [BddcSolver(p, precision="mixed").coarse_matrices(1) for p in probs]
    assert [max(k.shape[0] for k in kc) > 361 for kc in alone] == [True, True]
    errors = []

    def work(t):
        try:
            st = torch.cuda.Stream()
            for r in range(3):
                k = (t + r) % 2
                kc = BddcSolver(probs[k], precision="mixed", stream=st).coarse_matrices(1)
                for a, b in zip(kc, alone[k]):
                    np.testing.assert_array_equal(a, b)
        except Exception as e:   # surfaced below
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors


def test_mixed_coarse_matrices():
    # tolerance kappa_2(A_i) 2^-24 as in test_gpu_coarse.py: the FP32 factor's backward error
    p = _ball(12, 80, 0.3)
    d = Bddc(p).levels[0]
    kc = BddcSolver(p, precision="mixed").coarse_matrices(1)
    big = int(np.argmax([k.shape[0] for k in kc]))
    for s in (big, 0):
        K, C = d.K[s], d.maps.sub_C[s]
        ev = np.linalg.eigvalsh(K + float(np.mean(np.diag(K))) * C.T @ C)
        err = np.linalg.norm(kc[s] - d.KC[s]) / np.linalg.norm(d.KC[s])
        print(f"n_c {kc[s].shape[0]}: K_Ci relative error {err:.2e}, kappa 2^-24 = {ev[-1] / ev[0] * 2.0 ** -24:.2e}")
        assert err < max(ev[-1] / ev[0], 64.0) * 2.0 ** -24
