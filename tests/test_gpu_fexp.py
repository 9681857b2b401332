"""Near field of the FP64 form as float expansions (csrc/fexp.cuh, p2p_fexp.cuh)
against direct sums in long double, at the sizes where the staging (128
sources), the 32 runs, the two-target spans and the target groups of 32 have
their edges, and the limits beyond which leaves go to the FP64 kernel.

theta = 0 makes every pair pairwise.  Bounds, per component, in units of
A = sum_j |pair term| and with u = 2^-53: outside the kernels the expansions
are good to 2^-56 A and each flush adds one rounding, so 2^-50 A covers the
flushes of 512 sources, the far field and the final scaling; the FP64 kernel
and softened pairs carry the rounding of each term (the M4 polynomial cancels
by up to 120 near q = 2, which gives 120 x 8 u) and of a sum of n terms.
"""
import numpy as np
import pytest

from gpu_helpers import solver

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _m4(r, h):
    q = r / h
    L = np.longdouble
    with np.errstate(divide="ignore", invalid="ignore"):
        g = np.where(q < 1, (L(4) / 3 - L(6) / 5 * q**2 + q**3 / 2) / h**3,
                     (L(8) / 3 - 3 * q + L(6) / 5 * q**2 - q**3 / 6) / h**3 - 1 / (15 * r**3))
        p = np.where(q < 1, (-L(7) / 5 + L(2) / 3 * q**2 - L(3) / 10 * q**4 + q**5 / 10) / h,
                     (-L(8) / 5 + L(4) / 3 * q**2 - q**3 + L(3) / 10 * q**4 - q**5 / 30) / h + 1 / (15 * r))
        return np.where(q >= 2, 1 / r**3, g), np.where(q >= 2, -1 / r, p)


def _direct(pos, m, h):
    """Accelerations, potentials and the sums of absolute terms."""
    pos, m, h = (np.asarray(v, np.longdouble) for v in (pos, m, h))
    n = len(m)
    acc, pot = np.zeros((n, 3), np.longdouble), np.zeros(n, np.longdouble)
    A, B = np.zeros((n, 3), np.longdouble), np.zeros(n, np.longdouble)
    for i in range(n):
        d = pos[i] - np.delete(pos, i, 0)
        mj, hj = np.delete(m, i), np.delete(h, i)
        r = np.sqrt((d * d).sum(1))
        (gi, pi), (gj, pj) = _m4(r, h[i]), _m4(r, hj)
        t = (mj * (gi + gj) / 2)[:, None] * d
        acc[i], A[i] = -t.sum(0), np.abs(t).sum(0)
        pot[i], B[i] = (mj * (pi + pj) / 2).sum(), np.abs(mj * (pi + pj) / 2).sum()
    return acc, pot, A, B


def _set(n, seed, scale=1.0, shift=0.0):
    r = np.random.default_rng(seed)
    pos = r.uniform(-1, 1, (n, 3)) * scale + shift
    return pos, r.uniform(0.5, 1.5, n) / n, r


def _check(pos, m, h, leaf, bound, **opts):
    s = solver("fp64", **opts)
    s.build(pos, m, h, leaf)
    acc, pot = (t.cpu().numpy() for t in s.gravity(0.0, 0))
    s.close()
    a, p, A, B = _direct(pos, m, h)
    assert (np.abs(acc - a) <= bound * A + 1e-300).all(), float((np.abs(acc - a) / (A + 1e-300)).max() / U)
    assert (np.abs(pot - p) <= bound * B + 1e-300).all(), float((np.abs(pot - p) / (B + 1e-300)).max() / U)


@pytest.mark.parametrize("n,leaf", [(1, 16), (2, 1), (2, 16), (3, 2), (31, 32), (33, 64), (64, 64), (65, 64), (97, 33),
                                    (127, 16), (128, 10), (129, 7), (255, 64), (512, 16)])
def test_unsoftened_pairs(n, leaf):
    pos, m, r = _set(n, n + leaf)
    d = np.linalg.norm(pos[:, None] - pos[None], axis=2) + np.eye(n) * 9
    _check(pos, m, np.full(n, min(0.49 * d.min(), 0.5)), leaf, 2.0 ** -50)


@pytest.mark.parametrize("n,leaf,opts", [(2, 2, {}), (40, 64, {}), (129, 16, {}), (300, 12, {}), (300, 1, {"p2p_chunk": 32})])
@pytest.mark.parametrize("scale,shift", [(1.0, 0.0), (1e-9, 1.0), (3e40, 0.0)])
def test_softened_pairs(n, leaf, opts, scale, shift):
    pos, m, r = _set(n, 3 * n + leaf, scale, shift)
    _check(pos, m, scale * r.uniform(0.05, 0.6, n), leaf, (960 + n) * U, **opts)


@pytest.mark.parametrize("what", ["small h", "some small h", "masses", "far from the origin", "on the axes", "huge", "close pair",
                                  "close pair, tiny box"])
def test_limits(what):
    n = 200
    pos, m, r = _set(n, 77)
    h = np.full(n, 0.1)
    if what == "small h":
        h[:] = 1e-9
    elif what == "some small h":
        h[::17] = 1e-8
    elif what == "masses":
        m[::13] *= 1e-40
    elif what == "far from the origin":
        pos, h = pos + 1e7, h + 0.0
    elif what == "on the axes":
        pos[::3, 0] *= 1e-12
        pos[1::3, 1] = 0.0
    elif what.startswith("close pair"):
        # distinct particles with 1/r^3 beyond the largest double, well inside
        # their kernels: r = 1e-110 in a box of 1, 1e-104 in one of 1e-90
        s, r12 = (1e-90, 1e-104) if "tiny" in what else (1.0, 1e-110)
        pos, h = pos * s, h * s
        pos[0], pos[1] = 0.0, (r12, 0.0, 0.0)
    else:
        pos, h = pos * 1e95, h * 1e95
    _check(pos, m, h, 8, (960 + n) * U)


def test_systems_of_different_scales():
    from paper_2602_05804_gb300 import sfmm  # noqa: F401

    parts = [(_set(n, 5 + n, sc, sh), sc) for n, sc, sh in ((1, 1.0, 3.0), (90, 1e-6, 0.0), (140, 1e5, 1e6), (33, 1.0, 0.0))]
    pos = np.concatenate([p[0][0] for p in parts])
    m = np.concatenate([p[0][1] * 10.0 ** (3 * k) for k, p in enumerate(parts)])
    h = np.concatenate([np.full(len(p[0][1]), 0.2 * p[1]) for p in parts])
    off = np.concatenate([[0], np.cumsum([len(p[0][1]) for p in parts])])
    s = solver("fp64")
    s.build_batch(off, pos, m, h, np.full(4, 9, np.int32))
    acc, pot = (t.cpu().numpy() for t in s.gravity(0.0, 0))
    s.close()
    for a, b in zip(off[:-1], off[1:]):
        ra, rp, A, B = _direct(pos[a:b], m[a:b], h[a:b])
        assert (np.abs(acc[a:b] - ra) <= (960 + b - a) * U * A + 1e-300).all()
        assert (np.abs(pot[a:b] - rp) <= (960 + b - a) * U * B + 1e-300).all()


def _near_field_ms(pos, m, h, **opts):
    s = solver("fp64", profile=1, **opts)
    s.build(pos, m, h, 16)
    best = np.inf
    for _ in range(5):
        s.gravity(0.5, 2)
        best = min(best, s.stats()["ms_p2p"])
    s.close()
    return best


def test_items_left_to_fp64_fill_the_gpu():
    # far from the origin every item is left to the FP64 kernel: three blocks
    # per SM against one (0.86 of its time; equal while one was all it got)
    import workloads

    pos, m, h = workloads.plummer(100_000, 31)
    pos = pos + 1e7
    assert _near_field_ms(pos, m, h) <= 0.95 * _near_field_ms(pos, m, h, p2p_blocks=1)
