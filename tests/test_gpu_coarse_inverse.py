"""The dense coarsest inverse (blocked Gauss-Jordan on the device) and its transpose, on forests whose finest level is the
coarsest one (block edge 4), so that one cycle is u = A^-1 f.

Bound: with X the computed inverse, |A X f - f| <= c N eps cond(A) |f| for elimination with partial pivoting without element
growth (the operators are M-matrices up to the interface rows).  For k = 1 on an m^3 grid cond(A) = cot^2(pi / (2 m)) <
(2 m / pi)^2; a refined level doubles m.  c = 4."""
import math

import numpy as np
import pytest
import torch

from tests.helpers import one_refined_root

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def _uniform(R):
    return [(0, i, j, k) for k in range(R) for j in range(R) for i in range(R)]


# unknowns: 64 (four panels), 512, 960 (refined: probed column by column, non-symmetric), 1728, and 13824 (narrow panels)
@pytest.mark.parametrize("R,keys", [(1, _uniform(1)), (2, _uniform(2)), (2, one_refined_root()), (3, _uniform(3)),
                                    (6, _uniform(6))])
def test_direct_solve_and_its_transpose(R, keys):
    from paper_2403_08063_gb300 import Forest
    N = 64 * len(keys)
    F = Forest(R, 4, keys, max_coarse=N)
    assert F.levels() == [(len(keys), 4)]
    f = torch.from_numpy(np.random.default_rng(5).normal(size=(len(keys), 64))).cuda()
    F.set_rhs(f)
    u = torch.zeros_like(f)
    F.vcycle(u, 1)
    m = 4 * R * 2 ** max(key[0] for key in keys)
    bound = 4 * N * EPS * (2 * m / math.pi) ** 2
    assert float((F.apply(u) - f).norm() / f.norm()) <= bound
    if N <= 2000:  # the transpose, through the transposed cycle
        lam, _ = F.adjoint(u, f, want_k=False, rtol=bound * m, max_cycles=1)  # rtol in the volume-weighted norm
        assert float((F.apply_transpose(lam) - f).norm() / f.norm()) <= bound
    F.close()


def test_problems_with_different_unknowns():
    """A multi-problem level: one block, eight blocks and a refined problem side by side, each as if alone."""
    from paper_2403_08063_gb300 import Forest
    rows, starts = [], [0]
    problems = [[(0, 0, 0, 0)], [(1, i, j, k) for k in (0, 1) for j in (0, 1) for i in (0, 1)],
                [(1, i, j, k) for k in (0, 1) for j in (0, 1) for i in (0, 1) if (i, j, k) != (1, 0, 1)]
                + [(2, 2 + a, b, 2 + c) for c in (0, 1) for b in (0, 1) for a in (0, 1)]]
    for p, keys in enumerate(problems):
        rows += [(p, *key) for key in keys]
        starts.append(len(rows))
    f = torch.from_numpy(np.random.default_rng(6).normal(size=(len(rows), 64))).cuda()
    F = Forest(1, 4, np.array(rows, np.int32), n_problems=len(problems), max_coarse=2000)
    F.set_rhs(f)
    u = torch.zeros_like(f)
    F.vcycle(u, 1)
    for p, keys in enumerate(problems):
        G = Forest(1, 4, keys, max_coarse=2000)
        part = f[starts[p]:starts[p + 1]].contiguous()
        G.set_rhs(part)
        v = torch.zeros_like(part)
        G.vcycle(v, 1)
        assert torch.equal(v, u[starts[p]:starts[p + 1]])
        G.close()
    F.close()


def _dense(F, shape):
    """The operator's matrix, a column per unit vector."""
    n = shape[0] * shape[1]
    A = torch.empty((n, n), dtype=torch.float64, device="cuda")
    e = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for m in range(n):
        e.view(-1)[m] = 1.0
        A[:, m] = F.apply(e).view(-1)
        e.view(-1)[m] = 0.0
    return A


@pytest.mark.parametrize("R,sigma", [(1, 1.0), (2, 3.0), (3, 1.0)])
def test_direct_solve_with_rough_coefficients(R, sigma):
    """A symmetric, diagonally dominant operator (no interface) is eliminated without row exchanges: the bound above, with
    the condition number of the assembled matrix."""
    from paper_2403_08063_gb300 import Forest
    keys = _uniform(R)
    N, shape = 64 * len(keys), (len(keys), 64)
    rng = np.random.default_rng(7)
    F = Forest(R, 4, keys, coeff=True, max_coarse=N)
    f = torch.from_numpy(rng.normal(size=shape)).cuda()
    F.set_rhs(f, torch.from_numpy(np.exp(sigma * rng.normal(size=shape))).cuda())
    u = torch.zeros_like(f)
    F.vcycle(u, 1)
    s = torch.linalg.svdvals(_dense(F, shape).cpu())
    assert float((F.apply(u) - f).norm() / f.norm()) <= 4 * N * EPS * float(s[0] / s[-1])
    F.close()


def test_coefficients_beyond_binary64_contrast_are_still_accepted():
    """Two neighbouring cells of k = 2^66 among cells of k = 1: the other faces are lost in their diagonals, the second of the
    two has no diagonal pivot left, and the elimination exchanges rows as it does for other matrices."""
    from paper_2403_08063_gb300 import Forest
    keys = _uniform(1)
    k = torch.ones((1, 64), dtype=torch.float64, device="cuda")
    k[0, 21:23] = 2.0 ** 66
    F = Forest(1, 4, keys, coeff=True)
    F.set_rhs(torch.ones_like(k), k)
    u = torch.zeros_like(k)
    F.vcycle(u, 1)
    assert bool(torch.isfinite(u).all())
    k.fill_(1.0)  # and the next coefficients are inverted as usual
    F.set_rhs(torch.ones_like(k), k)
    u.zero_()
    F.vcycle(u, 1)
    assert float((F.apply(u) - 1.0).norm() / 8.0) <= 4 * 64 * EPS * (8 / math.pi) ** 2
    F.close()


def test_contrast_in_one_problem_leaves_its_neighbour_alone():
    """The same coefficients in a problem beside one with interfaces, whose pivots are searched for anyway."""
    from paper_2403_08063_gb300 import Forest
    refined = [(1, i, j, k) for k in (0, 1) for j in (0, 1) for i in (0, 1) if (i, j, k) != (1, 0, 1)]
    refined += [(2, 2 + a, b, 2 + c) for c in (0, 1) for b in (0, 1) for a in (0, 1)]
    rows = [(0, 0, 0, 0, 0)] + [(1, *key) for key in refined]
    k = torch.ones((len(rows), 64), dtype=torch.float64, device="cuda")
    k[0, 21:23] = 2.0 ** 66
    f = torch.from_numpy(np.random.default_rng(9).normal(size=(len(rows), 64))).cuda()
    F = Forest(1, 4, np.array(rows, np.int32), coeff=True, n_problems=2, max_coarse=2000)
    F.set_rhs(f, k)
    u = torch.zeros_like(f)
    F.vcycle(u, 1)
    assert bool(torch.isfinite(u).all())
    G = Forest(1, 4, refined, coeff=True, max_coarse=2000)
    G.set_rhs(f[1:].contiguous(), k[1:].contiguous())
    v = torch.zeros_like(f[1:])
    G.vcycle(v, 1)
    assert torch.equal(v, u[1:])
    F.close()
    G.close()


@pytest.mark.parametrize("cells,exponent", [("pair", 17.0), ("pair", 18.6), ("cube", 17.4), ("cube", 18.2),
                                            ("cube", 18.9), ("cube", 19.7)])
def test_pivots_lost_in_rounding_are_searched_for(cells, exponent):
    """A pair or a cube of cells coupled by about 10^exponent times what couples them to the rest, with coefficients that
    cancel to rounding noise instead of zero: such an operator is eliminated with row exchanges, bit for bit as beside a
    problem whose pivots cancel exactly and which therefore has all problems of its forest searched."""
    from paper_2403_08063_gb300 import Forest
    rng = np.random.default_rng(int(10 * exponent))
    k = np.exp(rng.normal(size=(2, 4, 4, 4)))
    if cells == "pair":
        k[0, 1, 1, 1:3] = 10.0 ** exponent * rng.uniform(1, 2, size=2)
    else:
        k[0, 1:3, 1:3, 1:3] = 10.0 ** exponent * rng.uniform(0.3, 3, size=(2, 2, 2))
    k[1] = 1.0
    k[1, 1, 1, 1:3] = 2.0 ** 66
    k = torch.from_numpy(k.reshape(2, 64)).cuda()
    f = torch.from_numpy(rng.normal(size=(2, 64))).cuda()
    got = []
    for problems in (1, 2):
        F = Forest(1, 4, [(p, 0, 0, 0, 0) for p in range(problems)], coeff=True, n_problems=problems)
        F.set_rhs(f[:problems].contiguous(), k[:problems].contiguous())
        u = torch.zeros_like(f[:problems])
        F.vcycle(u, 1)
        assert bool(torch.isfinite(u).all())
        got.append(u[0])
        F.close()
    assert torch.equal(got[0], got[1])


def test_narrow_panels_search_for_pivots():
    """More unknowns than one cluster's shared memory takes in panels of 16, with interfaces: panels of 4."""
    from paper_2403_08063_gb300 import Forest
    keys = one_refined_root(6)
    N = 64 * len(keys)
    F = Forest(6, 4, keys, max_coarse=N)
    f = torch.from_numpy(np.random.default_rng(8).normal(size=(len(keys), 64))).cuda()
    F.set_rhs(f)
    u = torch.zeros_like(f)
    F.vcycle(u, 1)
    assert float((F.apply(u) - f).norm() / f.norm()) <= 4 * N * EPS * (2 * 48 / math.pi) ** 2
    F.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_faces_averaged_beside_a_finer_interface(precision):
    """A refined root among 4^3: on the merged levels the two sides of its faces average different fine faces, so the
    coarsest operator has no interface and is not symmetric.  FP64 cycles against the oracle, and the mixed solve's residual."""
    import synthetic as syn
    from oracle.octree_mg import OracleMG
    from paper_2403_08063_gb300 import Forest
    R, n, keys = 4, 8, one_refined_root(4, (1, 2, 1))
    k = syn.lognormal_k_rff(R, n, keys, seed=51)
    f = syn.uniform_rhs(len(keys), n, seed=52)
    F = Forest(R, n, keys, coeff=True, precision=precision, coarse_coef="faces")
    F.set_rhs(f.cuda(), k.cuda())
    u = torch.zeros(f.shape, dtype=torch.float64, device="cuda")
    ref = OracleMG(R, n, keys, k_user=k.numpy(), coarse_coef="faces")
    if precision == 0:
        F.vcycle(u, 3)
        want, _ = ref.solve(f.numpy(), cycles=3)
        assert np.linalg.norm(u.cpu().numpy() - want) <= 1e-10 * np.linalg.norm(want)
    else:
        F.solve(u, rtol=1e-10)
        assert ref.rel_residual(u.cpu().numpy(), f.numpy()) <= 1.05e-10
    F.close()
