"""Kernels at the sizes where their tiling, splitting or number formats change.
Tolerances: FP64 results 1e-11 of the largest entry (a few thousand roundings
of 1.1e-16, amplified by at most the factor 2 k1 = 158 of the entropy); mixed
ones 1e-4 (B0), as everywhere in the suite."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h(vl):
    handle = vl.Handle(0)
    yield handle
    handle.close()


def _f64(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


# one pair; pairs just below, at and above one CTA of pairs (17 -> 136, 16 ->
# 120); fewer samples than a split's minimum; a spike beyond |u| = 22, where the
# fixed-point functions hand over to FP64
@pytest.mark.parametrize("m,n,spike", [(2, 2, 0), (2, 17, 0), (16, 15, 0), (17, 33, 0),
                                       (5, 1500, 30.0), (3, 6000, 75.0)])
def test_fp64_measure_sizes_and_outliers(vl, h, m, n, spike):
    rng = np.random.default_rng(m * 1000 + n)
    E = rng.laplace(size=(m, n))
    E[1:] += 0.4 * E[:-1]
    if spike:
        E[0, n // 2] = spike * E[0].std() * 1.5
        E[-1, 0] = -spike * E[-1].std()
    if n == 2:
        E[:, 1] = E[:, 0] + 1.0 + np.arange(m)  # |rho| = 1: degenerate
    Hx, Hr, D = _f64(m), _f64(m, m), _f64(m, m)
    vl.vl_pairwise_measure(h, torch.from_numpy(E).cuda(), "fp64", Hx, Hr, D)
    if n == 2:
        with pytest.raises(vl.VLError) as ei:
            h.sync()
        assert ei.value.code == 4  # VL_ERR_DEGENERATE
        return
    h.sync()
    ref = oracle.pairwise_measure(oracle.standardize(E))
    off = ~np.eye(m, dtype=bool)
    for got, want in ((Hx, ref["Ex"]), (Hr, np.where(off, ref["Er"], 0.0)), (D, ref["D"])):
        want = np.asarray(want)
        err = np.abs(got.cpu().numpy() - want)
        assert err.max() <= 1e-11 * max(1.0, np.abs(want).max())


# one cluster: the last block of 1, 31 and 32 rows, the chain alone (up to 96),
# one worker, seven, all of its range; beyond, the 64-wide blocks: last ones of
# 1, 63, 64 and 1 rows
@pytest.mark.parametrize("prec,m", [("mixed", m) for m in (2, 31, 32, 33, 64, 65, 96, 97, 128, 129,
                                                           320, 385, 511, 512, 513, 575, 576, 577)]
                         + [("fp64", m) for m in (513, 575, 576, 577)])
def test_fit_b_at_the_edges_of_the_factorisations(vl, h, prec, m):
    rng = np.random.default_rng(m)
    n = 2 * m + 7
    L = np.tril(rng.uniform(-0.4, 0.4, (m, m)) * (rng.random((m, m)) < 3.0 / m), -1)
    perm = rng.permutation(m)
    E = np.empty((m, n))
    E[perm] = np.linalg.solve(np.eye(m) - L, rng.laplace(size=(m, n)))
    order = torch.from_numpy(perm.astype(np.int32)).cuda()
    B0 = _f64(m, m)
    vl.vl_fit_b(h, torch.from_numpy(E).cuda(), order, None, prec, B0, None)
    h.sync()
    ref = oracle.fp64.b0_ldl(E, list(perm))
    assert np.abs(B0.cpu().numpy() - ref).max() <= (1e-4 if prec == "mixed" else 1e-10)


# tiles of the finalisation (7, 8, 9 variables); one and two exact segments of
# the tensor-core product (256 and 257 samples); standardized samples written in
# place and transposed (m n on either side of 2^19).  Variables 0 and 1 are nearly
# collinear (1 - rho^2 about 2.5e-3, where the pair constants take the FP64 form).
@pytest.mark.parametrize("m,n", [(7, 256), (8, 257), (9, 1000), (33, 15887), (33, 15889)])
def test_mixed_measure_at_the_edges_of_its_kernels(vl, h, m, n):
    rng = np.random.default_rng(m + n)
    E = rng.laplace(size=(m, n))
    E[2:] += 0.3 * E[:-2]
    E[1] = E[0] + 0.05 * rng.laplace(size=n)
    Hx, Hr, D = _f64(m), _f64(m, m), _f64(m, m)
    vl.vl_pairwise_measure(h, torch.from_numpy(E).cuda(), "mixed", Hx, Hr, D)
    h.sync()
    ref = oracle.pairwise_measure(oracle.standardize(E))
    off = ~np.eye(m, dtype=bool)
    want = np.where(off, ref["Er"], 0.0)
    # the suite's bounds for the mixed path: 1e-5 of the entropy scale and of max |D|
    assert np.abs(Hx.cpu().numpy() - ref["Ex"]).max() <= 1e-5 * max(1.42, np.abs(ref["Ex"]).max())
    assert np.abs(Hr.cpu().numpy() - want).max() <= 1e-5 * max(1.42, np.abs(want).max())
    assert np.abs(D.cpu().numpy() - ref["D"]).max() <= 1e-5 * np.abs(ref["D"]).max()


def _order_fp64(D):
    """Algorithm 1 with running FP64 sums: the order, each step's relative gap, and
    how far that gap may be off: the sums start from pairs of 48 bits and take m
    subtractions, so each score carries up to (m + 16) 2^-49 of its initial sum."""
    m = D.shape[0]
    P = np.minimum(D, 0.0) ** 2
    np.fill_diagonal(P, 0.0)
    S0 = P.sum(1)
    S, alive = S0.copy(), np.ones(m, dtype=bool)
    order, gap, slack = [], [], []
    for _ in range(m):
        left = np.flatnonzero(alive)
        by = left[np.argsort(S[left], kind="stable")[:2]]
        order.append(int(by[0]))
        gap.append(np.inf)
        slack.append(0.0)
        if len(by) == 2:
            a, b = P[np.ix_(by, left)].sum(1)
            gap[-1] = (b - a) / max(a, b, 1e-300)
            slack[-1] = 4 * (m + 16) * 2.0 ** -49 * S0[by].max() / max(a, b, 1e-300)
        alive[by[0]] = False
        S = S - P[:, by[0]]
    return order, np.array(gap), np.array(slack)


# the last size of each search (warps, variables per thread, where P is kept)
# and the first of the next
@pytest.mark.parametrize("m", [1, 31, 32, 33, 64, 65, 128, 129, 160, 161, 256, 257, 448, 449, 512,
                               513, 1024, 1025, 2048, 2049])
def test_order_at_the_edges_of_its_searches(vl, h, m):
    rng = np.random.default_rng(m)
    A = rng.normal(size=(m, m)) + 3.0 * rng.normal(size=m)[:, None]
    D = A - A.T
    if m > 40:  # not antisymmetric everywhere: both directions penalised
        D[3, 7] = D[7, 3] = -2.0
    order = torch.empty(m, dtype=torch.int32, device="cuda")
    gap = _f64(m)
    vl.vl_causal_order(h, torch.from_numpy(D).cuda(), order, gap)
    h.sync()
    want, want_gap, slack = _order_fp64(D)
    assert order.cpu().tolist() == want
    got = gap.cpu().numpy()
    assert np.array_equal(np.isinf(got), np.isinf(want_gap))
    fin = np.isfinite(want_gap)
    assert np.all(np.abs(got[fin] - want_gap[fin]) <= 1e-9 + slack[fin])


# lag windows: fewer samples than a block has threads, one more, ends of windows
# that fall to the first threads again, more lags than a warp and than a block.  A
# trend makes every window's mean a different one.  Tolerances: FP64 normal
# equations of condition up to 2e3, n 2.2e-16 each: 6.6e-10, taken as 1e-9; mixed
# 1e-5 (FP32 rounding of the series, 6e-8, by a condition of up to 160).
@pytest.mark.parametrize("m,n,p", [(3, 199, 1), (3, 256, 1), (3, 257, 2), (2, 259, 3),
                                   (2, 300, 40), (2, 513, 60), (2, 1500, 255), (2, 1500, 256)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_var_fit_with_different_window_means(vl, h, prec, m, n, p):
    if prec == "mixed" and p > 60:
        pytest.skip("condition beyond the tolerance's")
    rng = np.random.default_rng(n + p)
    X = rng.laplace(size=(m, n))
    for t in range(1, n):
        X[:, t] += 0.5 * X[:, t - 1]
    X += np.linspace(2.0, 5.0, n)
    M = _f64(p, m, m)
    vl.vl_var_fit(h, torch.from_numpy(X).cuda(), p, prec, M, None)
    h.sync()
    Z = np.vstack([np.ones(n - p)] + [X[:, p - b:n - b] for b in range(1, p + 1)]).T
    beta = np.linalg.lstsq(Z, X[:, p:].T, rcond=None)[0][1:]
    want = beta.reshape(p, m, m).transpose(0, 2, 1)
    tol = 1e-9 if prec == "fp64" else 1e-5
    assert np.abs(M.cpu().numpy() - want).max() <= tol


# the re-evaluated pairs of a certified ordering by one warp, two, four and eight:
# series just below and at the lengths where their number changes, odd ones among
# them.  The planted near tie is decided as by the exact measure, nothing left open.
@pytest.mark.parametrize("n", [121, 255, 256, 511, 512, 1023, 1024, 3001])
def test_certified_pairs_at_the_lengths_of_their_splits(vl, h, n):
    from test_gpu_parity import _planted_near_tie
    for seed in range(50):  # a tie whose planting swaps the two picks alone
        rng = np.random.default_rng(1000 * n + seed)
        E = rng.laplace(size=(12, n))
        for i in range(1, 12):
            E[i] += 0.6 * E[(i * 7) % i] + 0.4 * E[i - 1]
        D = np.asarray(oracle.pairwise_measure(oracle.standardize(E))["D"])
        od = oracle.order_heuristic(D)
        ref = [int(c) for c in od["order"]]
        Dp, k, a, b = _planted_near_tie(D, od["order"], od["steps"])
        swapped = ref[:k] + [b, a] + ref[k + 2:]
        if [int(c) for c in oracle.order_heuristic(Dp)["order"]] == swapped:
            break
    else:
        pytest.fail("no such series")
    order = torch.empty(12, dtype=torch.int32, device="cuda")
    stats = torch.zeros(4, dtype=torch.int32, device="cuda")
    vl.vl_causal_order_certified(h, torch.from_numpy(Dp).cuda(), torch.from_numpy(E).cuda(), order,
                                 None, stats)
    h.sync()
    assert [int(c) for c in order.cpu().numpy()] == ref
    st = [int(v) for v in stats.cpu().numpy()]
    assert st[1] >= 1 and st[2] >= 1 and st[3] == 0, st
