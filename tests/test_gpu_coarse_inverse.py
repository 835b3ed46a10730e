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
