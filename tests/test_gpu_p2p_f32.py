"""Near field of the FP32 form (csrc/p2p_f32.cuh) against direct sums, where
its staging (pairs of sources, 128 to a buffer), marks (32 steps a lane), result
windows (64) and target slots (32) have their edges, from no pair inside a
kernel to every one (a few marks are dealt over the lanes, more are evaluated
by the lanes that hold them, kernels far beyond the leaf take no marks), and h
below the normal FP32 range of (2h)^2.

theta = 0 makes every pair pairwise.  Bound per component, in units of A =
sum_j |pair term|: positions are FP32 offsets from leaf centres, so a
separation r is good to 2^-23 l / r with leaf size l (l / r < 10 here, the sets
keep a least distance), three times that for r^-3, plus 20 roundings of a term
and those of the sums: (3 x 2 x 10 + 20 + 30) 2^-24 < 7e-6."""
import numpy as np
import pytest

from gpu_helpers import solver

pytestmark = pytest.mark.gpu


def _m4(r, h):
    q = r / h
    g = np.where(q < 1, (4 / 3 - 1.2 * q**2 + q**3 / 2) / h**3,
                 (8 / 3 - 3 * q + 1.2 * q**2 - q**3 / 6) / h**3 - 1 / (15 * r**3))
    p = np.where(q < 1, (-1.4 + 2 / 3 * q**2 - 0.3 * q**4 + 0.1 * q**5) / h,
                 (-1.6 + 4 / 3 * q**2 - q**3 + 0.3 * q**4 - q**5 / 30) / h + 1 / (15 * r))
    return np.where(q >= 2, 1 / r**3, g), np.where(q >= 2, -1 / r, p)


@pytest.mark.parametrize("n,leaf", [(1, 16), (2, 16), (3, 2), (31, 32), (33, 33), (64, 64), (65, 64), (127, 16), (129, 7),
                                    (130, 64), (257, 31), (700, 11), (700, 1)])
@pytest.mark.parametrize("hs", ["none", "some", "uneven", "leaf", "all", "subnormal", "none at all"])
def test_direct_sum(n, leaf, hs):
    r = np.random.default_rng(7 * n + leaf)
    k = int(np.ceil(n ** (1 / 3)))
    grid = np.stack(np.meshgrid(*[np.arange(k)] * 3), -1).reshape(-1, 3)[:n] / k
    pos = grid + r.uniform(-0.3, 0.3, (n, 3)) / k
    m = r.uniform(0.5, 1.5, n) / n
    # in mean spacings of 1 / k: kernels of 2h below every distance, over about
    # ten neighbours, over fifty of one particle in 37 only, over a few leaves,
    # over the whole set; (2h)^2 below FLT_MIN; below FP32's least number
    h = {"none": 0.1, "some": r.uniform(0.4, 1.2, n), "uneven": np.where(np.arange(n) % 37 == 0, 1.2, 0.1),
         "leaf": r.uniform(2.0, 4.0, n), "all": 2.0 * k, "subnormal": 1e-21 * k, "none at all": 1e-300}[hs] / k * np.ones(n)
    s = solver("fp32")
    s.build(pos, m, h, leaf)
    acc, pot = (t.cpu().numpy() for t in s.gravity(0.0, 0))
    s.close()
    for i in range(n):
        d, mj, hj = pos[i] - np.delete(pos, i, 0), np.delete(m, i), np.delete(h, i)
        rr = np.sqrt((d * d).sum(1))
        with np.errstate(over="ignore", invalid="ignore"):
            (gi, pi), (gj, pj) = _m4(rr, h[i]), _m4(rr, hj)
        if hs == "none at all":
            gi = gj = 1 / rr**3
            pi = pj = -1 / rr
        t = (mj * (gi + gj) / 2)[:, None] * d
        u = mj * (pi + pj) / 2
        assert (np.abs(acc[i] + t.sum(0)) <= 7e-6 * np.abs(t).sum(0) + 1e-30).all()
        assert abs(pot[i] - u.sum()) <= 7e-6 * np.abs(u).sum() + 1e-30


def _per_pair(h, n=200_000):
    """Near-field time per pair of a set of n particles, least of five calls."""
    import workloads

    pos, m, _ = workloads.plummer(n, 21)
    s = solver("fp32", profile=1)
    s.build(pos, m, np.full(n, h), 16)
    best = np.inf
    for _ in range(6):
        s.gravity(0.5, 2)
        st = s.stats()
        best = min(best, st["ms_p2p"] / st["p2p_pairs"])
    s.close()
    return best


def test_kernels_beyond_the_leaves_cost_two_evaluations_a_pair():
    # a softened pair takes about 3 times an unsoftened one (6.5 times when each
    # was evaluated unsoftened, marked, dealt to a lane and handed back)
    assert _per_pair(0.2) <= 4.0 * _per_pair(1e-4)


def test_softening_as_good_as_none_costs_no_more():
    # every pair takes the unsoftened loops, whether (2h)^2 is a normal FP32
    # number or not (11 times the time when every pair was a marked one)
    assert _per_pair(1e-25) <= 1.5 * _per_pair(1e-4)
