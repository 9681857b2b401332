"""Paths that small sets and batches take: the one-block sort and scan at the
edges of their ranges (4096 particles, 8192 values), sums and boxes over slices
of a batch's systems, neighbour lists cut finer than the option when the lists
are few, FP64 moments translated a moment per lane where few lanes climb, and
the device memory that small sets and long lists take."""
import math

import numpy as np
import pytest

import oracle
import workloads
from gpu_helpers import TOL_FP64, acc_rel, pot_rel, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 31, 1023, 1024, 1025, 2049, 4095, 4096, 4097, 8191, 8192, 8193])
def test_sorted_order_and_tree(n):
    pos, m, h = workloads.plummer(n, 300 + n)
    pos[n // 3:n // 2] = pos[n // 3]  # equal keys: input order decides
    s = solver("fp32")
    s.build(pos, m, h, 8)
    t = s.tree()
    s.close()
    o = oracle.Tree(pos, m, h, 8, p=0)
    assert np.array_equal(t["perm"], o.perm)
    for k in ("first", "count", "right"):
        assert np.array_equal(t[k], getattr(o, k)), k


@pytest.mark.parametrize("sizes", [[6143], [6144], [6145], [22529], [150001], [2047, 1, 4097, 6144, 300]])
def test_sort_tiles(sizes):
    # tiles of 2048 keys, one per block, and the passes over the system index
    parts = [workloads.plummer(n, 70 + n) for n in sizes]
    for p in parts:
        n = len(p[1])
        p[0][n // 3:n // 2] = p[0][n // 3]
    off = np.concatenate([[0], np.cumsum(sizes)])
    pos, m, h = (np.concatenate([p[q] for p in parts]) for q in range(3))
    s = solver("fp32")
    s.build_batch(off, pos, m, h, np.full(len(sizes), 8, np.int32))
    perm = s.tree()["perm"]
    s.close()
    want = [a + oracle.Tree(*p, 8, p=0).perm for a, p in zip(off, parts)]
    assert np.array_equal(perm, np.concatenate(want))


def test_sums_of_sliced_systems():
    sizes = [1, 8191, 8192, 8193, 20001]
    parts = [workloads.plummer(k, 50 + k) for k in sizes]
    pos, m, h = (np.concatenate([p[q] for p in parts]) for q in range(3))
    off = np.concatenate([[0], np.cumsum(sizes)])
    s = solver("fp64")
    s.build_batch(off, pos, m, h, np.full(len(sizes), 8, np.int32))
    acc, pot = (t.cpu().numpy() for t in s.gravity(0.7, 1))
    sums, st = s.batch_sums(), s.stats()
    s.close()
    ma = m[:, None] * acc
    for k, (a, b) in enumerate(zip(off[:-1], off[1:])):
        for c in range(3):
            x = ma[a:b, c]
            assert abs(sums[k, c] - math.fsum(x)) <= 4e-16 * abs(math.fsum(x)) + 1e-25 * np.abs(x).sum()
        assert abs(sums[k, 3] - math.fsum(np.abs(ma[a:b]).ravel())) <= 1e-14 * sums[k, 3]
        assert abs(sums[k, 4] - 0.5 * math.fsum(m[a:b] * pot[a:b])) <= 1e-14 * abs(sums[k, 4])
    for c in range(3):
        assert abs(st["momentum"][c] - math.fsum(ma[:, c])) <= 4e-16 * abs(math.fsum(ma[:, c])) + 1e-25 * np.abs(ma).sum()
    assert abs(st["W"] - 0.5 * math.fsum(m * pot)) <= 1e-14 * abs(st["W"])


def _sums_batch(sizes):
    pos, m, h = workloads.plummer(int(sum(sizes)), 17)
    off = np.concatenate([[0], np.cumsum(sizes)])
    s = solver("fp32", profile=1)
    best = [np.inf, np.inf]
    for _ in range(4):
        s.build_batch(off, pos, m, h, np.full(len(sizes), 16, np.int32))
        acc, pot = s.gravity(0.8, 1)
        best = [min(best[0], s.stats()["ms_reduce"]), min(best[1], s.stats()["ms_build"])]
    out = s.batch_sums(), s.stats(), m[:, None] * acc.cpu().numpy(), m * pot.cpu().numpy(), off, best
    s.close()
    return out


def test_sums_of_one_large_system_among_small_ones():
    # slices of 8192 particles up to 64 of them, longer beyond; 1024 systems'
    # sums are added in a group
    r = np.random.default_rng(3)
    sizes = np.concatenate([r.integers(1, 12, 1500), [530_001], r.integers(1, 12, 18500)])
    sums, st, ma, mp, off, ms = _sums_batch(sizes)
    for k in list(range(0, len(sizes), 97)) + [1499, 1500, 1501, len(sizes) - 1]:
        a, b = off[k], off[k + 1]
        for c in range(3):
            x = math.fsum(ma[a:b, c])
            assert abs(sums[k, c] - x) <= 4e-16 * abs(x) + 1e-25 * np.abs(ma[a:b, c]).sum(), (k, c)
        assert abs(sums[k, 3] - np.abs(ma[a:b]).sum()) <= 1e-13 * sums[k, 3]
        assert abs(sums[k, 4] - 0.5 * mp[a:b].sum()) <= 1e-13 * np.abs(mp[a:b]).sum()
    for c in range(3):
        x = math.fsum(ma[:, c])
        assert abs(st["momentum"][c] - x) <= 4e-16 * abs(x) + 1e-25 * np.abs(ma).sum()
    assert abs(st["W"] - 0.5 * math.fsum(mp)) <= 1e-13 * abs(st["W"])
    # no system pays for the largest one (64 slices of the sums for each: 39
    # times, and 32 of the boxes: 3.6 times the build)
    even = _sums_batch(np.full(len(sizes), sizes.sum() // len(sizes)))[-1]
    assert ms[0] <= 6.0 * even[0]
    assert ms[1] <= 2.0 * even[1]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n,leaf", [(60, 4), (700, 16), (700, 64), (5000, 33), (3000, 1), (3000, 2), (2500, 7)])
def test_few_lists_are_cut_finer(prec, n, leaf):
    pos, m, h = workloads.binary_polytrope(n, 9)
    a_o, p_o, _ = oracle.sfmm(pos, m, h, theta=0.4, p=2, leaf_size=leaf)
    tol = TOL_FP64 if prec == "fp64" else 3e-5
    for chunk in (32, 65536):
        s = solver(prec, p2p_chunk=chunk)
        s.build(pos, m, h, leaf)
        acc, pot = (t.cpu().numpy() for t in s.gravity(0.4, 2))
        s.close()
        assert acc_rel(acc, a_o).max() <= tol and pot_rel(pot, p_o).max() <= tol


def test_leaves_of_one_are_not_cut_into_crumbs():
    # an item of 8 one-particle leaves costs its start and end: twice the time
    # of leaves of 16 (0.9 of it with 256 entries)
    pos, m, h = workloads.binary_polytrope(5000, 9)
    ms = []
    for leaf in (1, 16):
        s = solver("fp32", profile=1)
        s.build(pos, m, h, leaf)
        best = np.inf
        for _ in range(8):
            s.gravity(0.5, 2)
            best = min(best, s.stats()["ms_p2p"])
        ms.append(best)
        s.close()
    assert ms[0] <= 1.3 * ms[1], ms


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [700, 5000])
def test_blocks_per_sm_change_no_bit(prec, n):
    # where the lists are cut depends on the blocks that fit, not on those taken
    pos, m, h = workloads.plummer(n, 12)
    got = []
    for blocks in (0, 1, 2):
        s = solver(prec, p2p_blocks=blocks)
        s.build(pos, m, h, 16)
        got.append([t.cpu().numpy() for t in s.gravity(0.5, 2)])
        s.close()
    for a, p in got[1:]:
        np.testing.assert_array_equal(a, got[0][0])
        np.testing.assert_array_equal(p, got[0][1])


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_device_memory_of_small_sets(prec):
    # partial sums of cut lists are bounded by what the set's lists can hold: at
    # most a MB or two for 1000 particles (a bound by the GPU's size alone was
    # 120 MB more with leaves of 64 than a leaf size that cuts no list takes)
    import torch

    taken = []
    for leaf in (16, 64):
        pos, m, h = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in workloads.plummer(1000, 4))
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        s = solver(prec)
        s.build(pos, m, h, leaf)
        s.gravity(0.5, 2)
        taken.append(free - torch.cuda.mem_get_info()[0])
        s.close()
    assert abs(taken[1] - taken[0]) <= 16 << 20


@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("n,leaf", [(2, 1), (5, 1), (40, 1), (300, 2), (3000, 1), (20000, 16)])
def test_moments_of_the_climb(order, n, leaf):
    """The build's FP64 moments (warp-wide translation for up to four climbing
    lanes, a thread per node beyond) against the pass that translates every
    node by a thread: the same operations, so 1e-14 of the moments' scale
    leaves room for the leaf sums only."""
    pos, m, h = workloads.plummer(n, 60 + n)
    ref = solver("fp64")
    ref.build(pos, m, h, leaf)
    ref.gravity(0.8, 0)
    ref.build(pos, m, h, leaf)  # moments of order 0: the export makes its own
    Qr, mi = ref.moments(order)
    t = ref.tree()
    s = solver("fp64")
    s.build(pos, m, h, leaf)
    s.gravity(0.8, order)
    s.build(pos, m, h, leaf)  # moments of this order on the way up
    Q, _ = s.moments(order)
    ref.close()
    s.close()
    for k, deg in enumerate(np.asarray(mi).sum(1)):
        scale = t["mass"] * (t["size"] + 1e-16) ** deg + (1e-15 * t["mass"] if deg == 1 else 0.0)
        assert (np.abs(Q[:, k] - Qr[:, k]) <= 1e-14 * scale + 1e-30).all(), (order, k)


def test_walk_rings_grow_by_what_a_long_list_needs():
    """One kernel wider than the set: its leaf opens every other one, a list of
    more than 2^17 entries.  The rings of all resident warps then grow to 2^19
    entries (43 GB in the pair walk), not to 2^21 (172 GB)."""
    import torch

    pos, m, h = workloads.plummer(600_000, 6)
    h = h.copy()
    h[0] = 30.0
    pos, m, h = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (pos, m, h))
    torch.cuda.synchronize()
    got = []
    for sched in (3, 2):
        free = torch.cuda.mem_get_info()[0]
        s = solver("fp32", schedule=sched)
        s.build(pos, m, h, 4)
        got.append([t.cpu().numpy() for t in s.gravity(0.7, 1)])
        assert free - torch.cuda.mem_get_info()[0] <= 60e9
        s.close()
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])
