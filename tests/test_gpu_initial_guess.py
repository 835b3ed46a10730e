"""The start of a mixed-precision solve: a zero guess is not read again, any other is, wherever its values stand; and the
recorded cycles follow a changed launch shape and are counted like direct ones."""
import numpy as np
import pytest
import torch

import synthetic as syn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _forest(n, coeff=False, **kw):
    from paper_2403_08063_gb300 import Forest
    keys = [(0, i, j, k) for k in (0, 1) for j in (0, 1) for i in (0, 1)]
    F = Forest(2, n, keys, coeff=coeff, precision=1, **kw)
    f = syn.uniform_rhs(8, n, seed=71).to(DEV)
    k = syn.lognormal_k_rff(2, n, keys, seed=72, sigma=0.5, ell=0.3).to(DEV) if coeff else None
    F.set_rhs(f, k)
    return F, f


@pytest.mark.parametrize("n", [8, 32])
@pytest.mark.parametrize("at", [0.0, 0.5, 1.0])
def test_one_nonzero_value_of_the_guess_counts(n, at):
    """One value of 1e6 times the solution: a V-cycle divides it by 10 to 100, so the iterate stays far off."""
    F, f = _forest(n)
    sol = torch.zeros_like(f)
    F.solve(sol, rtol=1e-11)
    u = torch.zeros_like(f)
    u.view(-1)[int(at * (f.numel() - 1))] = 1e6 * float(sol.abs().max())
    rel = F.vcycle(u, 1)
    assert float((u - sol).norm()) > float(sol.norm())
    got = float((f - F.apply(u)).norm() / f.norm())
    assert got > 1.0 and abs(got - rel) <= 1e-6 * got
    F.close()


@pytest.mark.parametrize("coeff", [False, True])
def test_a_problem_without_a_right_hand_side_stays_at_zero(coeff):
    from paper_2403_08063_gb300 import Forest
    n = 8
    leaves = [(p, 0, 0, 0, 0) for p in range(3)]
    f = syn.uniform_rhs(3, n, seed=73).to(DEV)
    f[1] = 0.0
    k = torch.exp(0.3 * syn.uniform_rhs(3, n, seed=74)).to(DEV) if coeff else None
    F = Forest(1, n, leaves, coeff=coeff, precision=1)
    F.set_rhs(f, k)
    u = torch.zeros_like(f)
    F.solve(u, rtol=1e-10)
    assert torch.equal(u[1], torch.zeros_like(u[1]))
    r = f - F.apply(u)
    for p in (0, 2):
        # the recomputed residual differs from the solver's by rounding, eps * |A| |u| / |f| < 1e-12 here
        assert float(r[p].norm()) <= 1.02e-10 * float(f[p].norm())
    F.close()


@pytest.mark.parametrize("coeff", [False, True])
def test_recorded_cycles_follow_a_new_launch_shape_and_are_counted(coeff):
    F, f = _forest(32, coeff, inner_cycles=1)
    F.set_tail(-1)
    runs = []
    for shape in F.smoother_shapes(0)[:3]:
        F.set_smoother_shape(0, shape)
        for _ in range(3):  # direct, recorded, replayed
            u = torch.zeros_like(f)
            F.vcycle(u, 2)
            runs.append(u)
    for u in runs[1:]:
        assert torch.equal(u, runs[0])
    counts = []
    for timed in (True, False):  # a profiled run launches directly; the counters start at mg_profile(1)
        F.profile(True)
        F.profile(timed)
        F.vcycle(torch.zeros_like(f), 2)
        counts.append({name: v[1] for name, v in F.profile_read().items()})
    assert counts[0] == counts[1] and counts[0]["smooth_f32_finest"] > 0
    assert np.isfinite(float(runs[0].norm()))
    F.close()


@pytest.mark.parametrize("n", [4, 8, 16, 64])
@pytest.mark.parametrize("what", ["dense", "blocks", "last"])
def test_a_guess_is_read_and_written_once(n, what):
    """One layout launch packs a guess without a zero part (and one unpacks the result); parts that are zero are cleared of
    what an earlier solve left there.  The iterate is that of a forest that has solved nothing."""
    guess = torch.rand((8, n ** 3), generator=torch.Generator().manual_seed(75), dtype=torch.float64).to(DEV) + 0.5
    if what == "blocks":
        guess[::2] = 0.0
    elif what == "last":
        guess.view(-1)[:-1] = 0.0
    out = []
    for used in (False, True):
        F, f = _forest(n, inner_cycles=2)
        if used:
            F.solve(torch.zeros_like(f), rtol=1e-8)
        u = guess.clone()
        F.profile(True)
        rel = F.vcycle(u, 2)
        assert F.profile_read()["layout"][1] == (2 if what == "dense" else 3)
        F.profile(False)
        out.append((rel, u))
        F.close()
    assert out[0][0] == out[1][0] and torch.equal(out[0][1], out[1][1])
