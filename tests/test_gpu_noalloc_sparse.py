"""ttcross_sampled_error_noalloc on cores whose terms have scales of their own: sums
of TTs (block-diagonal middle cores) and CP forms (diagonal ones) with one block
2^t up in one core and down again in the next, a peak of 2^t that no sample hits,
entries that are subnormal, infinite or not numbers.  Fixed point relative to the
largest term would lose the other terms; every sample has to come out as exact as
its FP64 chain.

Tolerance: all entries are positive, so the chain of up to 5 cores of up to 32
terms is off by less than 5 * 32 * 2^-53 = 1.8e-14 of X~ itself (powers of two are
exact), and the error within less than that relative to itself, X~ being larger
than X: 1e-13."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

NS, SEED = 20000, 5


@pytest.fixture(scope="module")
def err():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross
    out = torch.zeros(1, dtype=torch.float64, device="cuda")

    def run(n, cores):
        ttcross.sampled_error_noalloc(n, {"kind": "hilbert"},
                                      [torch.from_numpy(c).cuda() for c in cores], NS, SEED, out)
        return out.item()
    return run


def reference(n, cores):
    idx = oracle.sample_indices(n, NS, SEED)
    x = (1.0 / (1.0 + idx.sum(axis=1))).astype(np.longdouble)
    v = cores[0].astype(np.longdouble)[0, idx[:, 0], :]
    for m in range(1, len(n)):
        c = cores[m].astype(np.longdouble)
        v = np.concatenate([np.einsum("sp,psq->sq", v[i:i + 1024], c[:, idx[i:i + 1024, m], :])
                            for i in range(0, NS, 1024)])
    return float(np.sqrt(((x - v[:, 0]) ** 2).sum() / (x ** 2).sum()))


def blocks(n, sizes, rng):
    """The cores of a sum of TTs of ranks ``sizes``, entries in [0.5, 1.5]."""
    r, d, cores = sum(sizes), len(n), []
    for m in range(d):
        c = np.zeros((1 if m == 0 else r, n[m], 1 if m == d - 1 else r))
        at = 0
        for s in sizes:
            p, q = slice(None) if m == 0 else slice(at, at + s), slice(None) if m == d - 1 else slice(at, at + s)
            c[p, :, q] = 0.5 + rng.random(c[p, :, q].shape)
            at += s
        cores.append(c)
    return cores


@pytest.mark.parametrize("t", [20, 70, 300])
@pytest.mark.parametrize("n,sizes,core", [
    ([20, 30, 40], [1, 1], 1),
    ([20, 30, 40], [3, 5], 1),
    ([20, 30, 40], [1] * 12, 1),                     # CP
    ([24, 33, 64, 48, 20], [9, 4], 1),
    ([24, 33, 64, 48, 20], [2, 13], 3),
    ([24, 33, 64, 48, 20], [17, 15], 2),
])
def test_blocks_of_other_scales(err, n, sizes, core, t):
    cores = blocks(n, sizes, np.random.default_rng(sum(n) + sum(sizes)))
    cores[core][:sizes[0]] *= 2.0 ** t
    cores[core + 1][:sizes[0]] *= 2.0 ** -t
    ref = reference(n, cores)
    got = err(n, cores)
    assert abs(got - ref) <= 1e-13 * ref, (got, ref)


@pytest.mark.parametrize("t", [40, 70, 300])
@pytest.mark.parametrize("n,r", [([20, 30, 40], 7), ([20, 30, 10, 25], 20)])
def test_peak_that_no_sample_hits(err, n, r, t):
    cores = blocks(n, [r, 1], np.random.default_rng(r))
    idx = oracle.sample_indices(n, NS, SEED)
    hit = set(map(tuple, idx))
    # shares all but its last index with samples
    peak = next(tuple(i[:-1]) + (j,) for i in idx for j in range(n[-1]) if tuple(i[:-1]) + (j,) not in hit)
    for m, c in enumerate(cores):
        row, col = (0 if m == 0 else r), (0 if m == len(n) - 1 else r)
        c[row, :, col] = 0.0
        c[row, peak[m], col] = 2.0 ** t if m == 1 else 1.0
    ref = reference(n, cores)
    got = err(n, cores)
    assert abs(got - ref) <= 1e-13 * ref, (got, ref)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("core", [0, 1, 2, 3])
def test_not_finite_as_the_chains_have_it(err, bad, core):
    n = [20, 30, 40, 16]
    cores = blocks(n, [7], np.random.default_rng(1))
    cores[core][0, 5, 0] = bad
    np.testing.assert_equal(err(n, cores), reference(n, cores))


def test_subnormal_entries(err):
    n = [20, 30, 40]
    rng = np.random.default_rng(2)
    sz = [1, 6, 5, 1]
    cores = [rng.integers(1, 9, (sz[m], n[m], sz[m + 1])).astype(float) for m in range(3)]
    plain = err(n, cores)
    for c, e in zip(cores, (-1060, 1000, 60)):
        c *= 2.0 ** (e / 2)
        c *= 2.0 ** (e / 2)
    assert err(n, cores) == plain
