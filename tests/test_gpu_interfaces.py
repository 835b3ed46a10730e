"""Interface ghosts, their transpose and the FP64 transfers at the block edges where the kernels change how they split
the work (one strip per interface face up to 16^2 cells, several from 32^2 on; the smallest block and the largest), against the
oracle on one root whose eighth octant is refined.  Bounds as in the other operator and cycle tests: 1e-13 for single
operators and exchanges (rounding of sums of at most 27 terms), 1e-10 relative for FP64 iterates."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle.octree_mg import OracleMG

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _octant():
    keys = [(1, i, j, k) for i in (0, 1) for j in (0, 1) for k in (0, 1) if (i, j, k) != (0, 1, 0)]
    return keys + [(2, i, 2 + j, k) for i in (0, 1) for j in (0, 1) for k in (0, 1)]


@pytest.mark.parametrize("n,coeff,variant", [(4, True, "C"), (4, False, "P"), (16, True, "C"), (32, False, "C"), (32, True, "P"),
                                             (64, True, "C"), (64, False, "P"), (128, True, "C")])
def test_interface_operators_match_oracle(n, coeff, variant):
    from paper_2403_08063_gb300 import Forest
    keys = _octant()
    rng = np.random.default_rng(n)
    shape = (len(keys), n ** 3)
    k = np.exp(0.5 * rng.normal(size=shape)) if coeff else None
    F = Forest(1, n, keys, coeff=coeff, interface_flux=variant == "C")
    F.set_rhs(torch.ones(shape, dtype=torch.float64, device=DEV), torch.from_numpy(k).to(DEV) if coeff else None)
    ref = OracleMG(1, n, keys, k_user=k, variant=variant, operator_only=True)
    u = rng.normal(size=shape)
    ud = torch.from_numpy(u).to(DEV)

    L = ref.levels[0]
    perm = [L.index[key] for key in F.level_keys(0)]
    block_of = {key: b for b, key in enumerate(keys)}
    rows = [block_of[key] for key in F.level_keys(0)]
    Uo = L.zeros()
    for b, ob in enumerate(perm):
        Uo[ob, 1:-1, 1:-1, 1:-1] = u[rows[b]].reshape(n, n, n)
    padded = F.exchange_level(0, ud[rows].contiguous()).cpu().numpy()
    ref.exchange(0, Uo)
    for axis in range(3):
        for side in (0, 1):
            sl = [slice(None), slice(1, -1), slice(1, -1), slice(1, -1)]
            sl[3 - axis] = (n + 1) * side
            got, want = padded[tuple(sl)], Uo[perm][tuple(sl)]
            assert np.abs(got - want).max() <= 1e-13 * np.abs(Uo).max(), (axis, side)

    got, want = F.apply(ud).cpu().numpy(), ref.apply_A(u)
    assert np.linalg.norm(got - want) <= 1e-13 * np.linalg.norm(want)
    got, want = F.apply_transpose(ud).cpu().numpy(), ref.apply_AT(u)
    assert np.linalg.norm(got - want) <= 1e-13 * np.linalg.norm(want)
    F.close()


@pytest.mark.parametrize("n,coeff,coarse_coef", [(128, True, "faces"), (128, False, "k")])
def test_fp64_cycles_on_the_largest_block(n, coeff, coarse_coef):
    """One 128^3 root down to 8^3: the FP64 restriction and prolongation at every edge they are written for."""
    from paper_2403_08063_gb300 import Forest
    keys = [(0, 0, 0, 0)]
    f = syn.uniform_rhs(1, n, seed=5)
    k = syn.lognormal_k_rff(1, n, keys, seed=6, sigma=0.5, ell=0.3) if coeff else None
    F = Forest(1, n, keys, coeff=coeff, coarse_coef=coarse_coef)
    F.set_rhs(f.to(DEV), k.to(DEV) if coeff else None)
    u = torch.zeros(f.shape, dtype=torch.float64, device=DEV)
    F.vcycle(u, 2)
    ref = OracleMG(1, n, keys, k_user=k.numpy() if coeff else None, coarse_coef=coarse_coef)
    want, _ = ref.solve(f.numpy(), cycles=2)
    assert np.linalg.norm(u.cpu().numpy() - want) <= 1e-10 * np.linalg.norm(want)
    F.close()
