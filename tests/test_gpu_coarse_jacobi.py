"""The coarsest level's damped Jacobi sweeps in one cluster launch, against the oracle: one block, one block per CTA, several
per CTA and CTAs without one; an odd and an even number of sweeps; constant and variable coefficients; and the level that
is both the finest and the coarsest.  Bound as in the other FP64 cycle tests: 1e-10 relative."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle.octree_mg import OracleMG

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,n,coeff,iters", [(1, 8, False, 7), (1, 8, True, 16), (2, 8, True, 33), (2, 8, False, 1),
                                             (3, 8, False, 40), (3, 8, True, 5), (3, 4, True, 64)])
def test_coarse_jacobi_sweeps_match_the_oracle(R, n, coeff, iters):
    from paper_2403_08063_gb300 import Forest
    keys = [(0, i, j, k) for k in range(R) for j in range(R) for i in range(R)]
    f = syn.uniform_rhs(len(keys), n, seed=31)
    k = syn.lognormal_k_rff(R, n, keys, seed=32, sigma=0.5, ell=0.3) if coeff else None
    F = Forest(R, n, keys, coeff=coeff, smoother="jacobi", omega=0.8, nu1=2, nu2=1, coarse_iters=iters)
    F.set_rhs(f.cuda(), k.cuda() if coeff else None)
    u = torch.zeros(f.shape, dtype=torch.float64, device="cuda")
    F.vcycle(u, 3)
    # a one-level forest sweeps on from its iterate (every release has), where the oracle's coarsest solve starts from zero:
    # three cycles there are one of three times the sweeps
    one = n == 4
    ref = OracleMG(R, n, keys, k_user=k.numpy() if coeff else None, nu1=2, nu2=1, smoother="jacobi", omega=0.8,
                   coarse_iters=3 * iters if one else iters)
    want, _ = ref.solve(f.numpy(), cycles=1 if one else 3)
    assert np.linalg.norm(u.cpu().numpy() - want) <= 1e-10 * np.linalg.norm(want)
    F.close()
