"""The size of a batch decides which kernel and how many lanes, warps or CTAs a
matrix gets, never its result: every row of a large batch equals, bit for bit,
the same matrix in a call on a few, across the sizes where the routes change;
sampled rows against the CPU oracle (tolerance 1e-10 times the sum of the
absolute values of the terms)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2104_07638_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.fixture(scope="module")
def apm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_07638_gb300 import apm as m
    m.lib()
    m.tune_set(None)
    m.tune_options_set(0, 0, 0)
    return m


def mixed(n, batch, seed):
    """Gaussian and Hubbard matrices; among the first ones zero diagonals (a
    correction at every pivot), equal vertices, the zero matrix, non-finite entries."""
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((batch, n, n))
    A[::2] = I.hubbard_batch(batch, n, seed=seed)[::2]
    A[1][np.diag_indices(n)] = 0.0
    A[3] = 0.0
    A[5, 0, n - 1] = np.inf
    A[7, n - 1, 0] = np.nan
    if n > 2:
        A[2][:, 1] = A[2][:, n - 1]
        A[2][1] = A[2][n - 1]
    return A


def rows_equal(big, small, idx):
    for x, y in zip(big, small):
        x, y = x[idx].cpu().numpy(), y.cpu().numpy()
        assert np.array_equal(x, y, equal_nan=True)


# both sides of every change of route and of CTA width at orders 1..11
LANES = [(1, 40), (2, 3000), (3, 40000), (4, 455), (4, 457), (4, 8000), (4, 30001), (5, 913), (5, 1501), (5, 3001),
         (5, 29200), (6, 2201), (6, 8001), (6, 14600), (6, 29190), (7, 4999), (7, 5501), (7, 20001), (8, 913),
         (8, 10001), (8, 20001), (9, 457), (9, 913), (10, 500), (10, 1000), (10, 1673), (11, 460)]


@pytest.mark.parametrize("n,batch", LANES)
def test_small_orders(apm, n, batch):
    A = mixed(n, batch, 8100 + n)
    B = I.hubbard_batch(batch, n, seed=8200 + n)
    d, e = torch.as_tensor(A).cuda(), torch.as_tensor(B).cuda()
    few = torch.as_tensor([0, 1, 2, 3, 5, 7, batch // 2, batch - 2, batch - 1]).cuda()
    for f in (lambda x, y: apm.cdet_connected(x, return_minors=True, return_status=True),
              lambda x, y: apm.cdet_connected(x, y, return_minors=True, return_status=True),
              lambda x, y: apm.cdet_connected(x, single_det=True, return_status=True, piv_threshold=0.5),
              lambda x, y: apm.all_minors(x, return_status=True)):
        rows_equal(f(d, e), f(d[few], e[few]), few)
    w = torch.as_tensor(np.random.default_rng(n).standard_normal((batch, 1 << n))).cuda()
    w[3, 0] = float("nan")                      # a[0] is not read
    rows_equal((apm.cdet_from_weights(w),), (apm.cdet_from_weights(w[few]),), few)
    c, m = apm.cdet_connected(d, return_minors=True)
    pick = [0, 1, 2, batch - 1]
    mref, ms = oracle.minors_lu(A[pick]), oracle.minors_scale(A[pick])
    assert np.all(np.abs(m.cpu().numpy()[pick] - mref) <= TOL * np.maximum(ms, 1e-300))
    cref, cs = oracle.cdet_recursion(mref * mref), oracle.cdet_scale(ms * ms)
    assert np.all(np.abs(c.cpu().numpy()[pick] - cref) <= TOL * np.maximum(cs, 1e-300))


# the warp-per-run minors kernel: tails of 9..12 elements, one run or several per matrix
@pytest.mark.parametrize("n,batch", [(9, 700), (10, 305), (11, 160), (11, 700), (12, 80), (12, 160), (12, 5000),
                                     (13, 39), (13, 5000), (14, 155), (15, 77), (16, 45)])
def test_minors_runs(apm, n, batch):
    d = torch.as_tensor(mixed(n, batch, 8300 + n)).cuda()
    few = torch.as_tensor([0, 1, 2, 3, 5, 7, batch // 2, batch - 2, batch - 1]).cuda()
    big, st = apm.all_minors(d, return_status=True)
    one = [apm.all_minors(d[i:i + 1].clone(), return_status=True) for i in few.tolist()]
    rows_equal((big, st), (torch.cat([m for m, _ in one]), torch.cat([s for _, s in one])), few)
    rows_equal((big, st), apm.all_minors(d[few], return_status=True), few)
    if n > 12:      # the connected sums' minors take the same route
        rows_equal((big[few], st[few]), apm.cdet_connected(d[few], return_minors=True, return_status=True)[1:],
                   list(range(9)))


# above order 12: one CTA per matrix, or the blocks of a matrix on many CTAs with
# the terms in rows of their own (few matrices) or summed in place, and the last
# partial round of a larger batch
@pytest.mark.parametrize("n,batch", [(13, 261), (13, 470), (14, 351), (14, 300), (15, 120), (15, 11)])
def test_blocked_orders(apm, n, batch):
    d = torch.as_tensor(mixed(n, batch, 8400 + n)).cuda()
    e = torch.as_tensor(I.hubbard_batch(batch, n, seed=8500 + n)).cuda()
    few = torch.as_tensor([0, 1, 2, 5, batch // 2, batch - 1]).cuda()
    for f in (lambda x, y: apm.cdet_connected(x, return_minors=True, return_status=True),
              lambda x, y: apm.cdet_connected(x, single_det=True, return_status=True),
              lambda x, y: apm.cdet_connected(x, y, return_minors=True, return_status=True)):
        rows_equal(f(d, e), f(d[few], e[few]), few)


@pytest.mark.parametrize("n,batch", [(13, 300), (14, 360), (16, 40)])
def test_blocked_orders_from_weights(apm, n, batch):
    w = torch.as_tensor(np.random.default_rng(n).standard_normal((batch, 1 << n))).cuda()
    few = torch.as_tensor([0, 3, batch // 2, batch - 1]).cuda()
    w[3, 0] = float("nan")                      # a[0] is not read
    c = apm.cdet_from_weights(w)
    rows_equal((c,), (apm.cdet_from_weights(w[few]),), few)
    # in place, as the one-CTA-per-matrix route takes it
    z = w[few].clone()
    nb = apm.workspace_size(apm.OP_CDET_FROM_WEIGHTS, n, 4)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    apm._check(apm.lib().apm_cdet_from_weights(apm._ptr(z), n, 4, apm._ptr(z), apm._ptr(ws), nb, apm._stream(z)),
               "apm_cdet_from_weights")
    rows_equal((c,), (z,), few)


# the fast subset convolution: rounds of one CTA per row, the last one by tiles
@pytest.mark.parametrize("n,batch", [(10, 500), (12, 520), (12, 530), (13, 460), (14, 457), (16, 459)])
def test_fast_subset_convolution(apm, n, batch):
    w = torch.rand((batch, 1 << n), dtype=torch.float64, device="cuda",
                   generator=torch.Generator(device="cuda").manual_seed(n))
    few = torch.as_tensor([0, 3, 455, 456, batch - 1]).cuda()
    rows_equal((apm.cdet_from_weights_fsc(w),), (apm.cdet_from_weights_fsc(w[few]),), few)


# two-spin Keldysh sums: pairs whole or split over warps (a rounding apart), one
# warp per CTA up to twelve, and scratch sized for a batch serving a smaller one
@pytest.mark.parametrize("n,batch", [(7, 40), (8, 304), (8, 305), (9, 77), (10, 153), (8, 1825)])
def test_keldysh2_splits(apm, n, batch):
    Mu, Md = (torch.as_tensor(x).cuda() for x in I.keldysh2_batch(batch, n, seed=8600 + n))
    Mu[3, 0, 1] = float("nan")
    s, p, st = apm.keldysh2_sum(Mu, Md, partial=True, return_status=True)
    few = [0, 1, 3, batch // 2, batch - 1]
    sf, pf, stf = apm.keldysh2_sum(Mu[few], Md[few], partial=True, return_status=True)
    assert torch.equal(st[few], stf) and int(stf[2]) == apm.ST_NONFINITE_INPUT
    good = [i for i in few if i != 3]
    scale = oracle.keldysh2_scale(Mu[good].cpu().numpy(), Md[good].cpu().numpy())
    at = [k for k, i in enumerate(few) if i != 3]
    assert np.all(np.abs((s[good] - sf[at]).cpu().numpy()) <= TOL * scale)
    assert np.all(np.abs((p[good] - pf[at]).cpu().numpy()) <= TOL * scale[:, None])
    assert bool(torch.isnan(s[3].real)) and bool(torch.isnan(pf[2].real).all())
    sizes = [apm.workspace_size(apm.OP_KELDYSH2, n, b) for b in (1, 76, 152, 305, 608, 1824, 4000)]
    assert sizes == sorted(sizes)


# XNOR minors and the Nambu connected sums: tails of 5, 7 and 8 vertices, whole
# matrices or runs of leaves; a singular block in one run makes the whole row NaN
@pytest.mark.parametrize("n,batch", [(10, 230), (10, 500), (10, 2000), (11, 120), (13, 30), (13, 60)])
def test_xnor_runs(apm, n, batch):
    M = I.nambu_batch(batch, n, seed=8700 + n)
    M[1, 2 * n - 2:, 2 * n - 2:] = 0.0            # met by the leaves that keep the last vertex
    M[2, 0, 3] = np.inf
    d = torch.as_tensor(M).cuda()
    few = torch.as_tensor([0, 1, 2, batch // 2, batch - 1]).cuda()
    big = apm.nambu_cdet(d, return_minors=True, return_status=True)
    rows_equal(big, apm.nambu_cdet(d[few], return_minors=True, return_status=True), few)
    st = big[2].cpu().numpy()
    assert st[1] == apm.ST_ZERO_PIVOT and st[2] == apm.ST_NONFINITE_INPUT and st[0] == 0 and not st[3:].any()
    assert bool(torch.isnan(big[1][1]).all()) and bool(torch.isnan(big[1][2]).all())
    assert not bool(torch.isnan(big[1][0]).any())
    sizes = [apm.workspace_size(apm.OP_XNOR_MINORS, n, b) for b in (1, 28, 113, 228, 456, 912, 1520, 5000)]
    assert sizes == sorted(sizes)


# two vertex types: the first pass whole (large batches) or by kept sets of the
# upper vertices, with a small pivot (redone), a singular and a non-finite matrix
@pytest.mark.parametrize("n,batch", [(7, 900), (7, 2500), (8, 1500), (9, 60), (10, 33)])
def test_two_type_parts(apm, n, batch):
    M = I.two_type_batch(batch, n, seed=8800 + n)
    M[1][np.diag_indices(2 * n)] = 0.0
    M[2, 1, 2] = np.inf
    M[4, 2 * n - 1, 2 * n - 1] = 0.0
    d = torch.as_tensor(M).cuda()
    few = torch.as_tensor([0, 1, 2, 3, 4, batch // 2, batch - 1]).cuda()
    for kw in ({}, {"piv_shift": 0.0}):          # no shift leaves a zero pivot flagged
        big = apm.two_type_cdet(d, return_weights=True, return_status=True, **kw)
        rows_equal(big, apm.two_type_cdet(d[few], return_weights=True, return_status=True, **kw), few)
        st = big[2].cpu().numpy()
        assert st[2] == apm.ST_NONFINITE_INPUT and bool(torch.isnan(big[1][2]).all()) and st[0] == 0
        assert (st[1] & apm.ST_ZERO_PIVOT) if kw else (st[1] & apm.ST_PIVOT_CORRECTED)
    if n <= 8:
        rows_equal(apm.nand_minors(d, return_status=True), apm.nand_minors(d[few], return_status=True), few)
    sizes = [apm.workspace_size(apm.OP_TWO_TYPE_CDET, n, b) for b in (1, 100, 1000, 4096, 4097, 20000)]
    assert sizes == sorted(sizes)


# an uneven batch of few items (orders 13..15 by blocks on many CTAs), of many, and
# fixed-order calls of the same matrices, with flagged ones among them
def test_uneven_few_and_many(apm):
    rng = np.random.default_rng(8900)
    few = np.concatenate([[15, 13, 16, 14, 15, 13, 14], rng.integers(4, 17, 60)]).astype(np.int32)
    many = np.concatenate([few, rng.integers(4, 13, 1100)]).astype(np.int32)
    flat, off = I.hubbard_varlen(many, seed=8901)
    flat[off[1]:off[1] + 169] = 0.0                     # redone with corrections
    flat[off[3]] = np.nan                               # non-finite
    A, ao, nt = (torch.as_tensor(x).cuda() for x in (flat, off, many))
    cm, mm, sm = apm.cdet_connected_varlen(A, ao, nt, return_minors=True, return_status=True)
    cf, mf, sf = apm.cdet_connected_varlen(A, ao[:few.size].contiguous(), nt[:few.size].contiguous(),
                                           return_minors=True, return_status=True)
    assert np.array_equal(cm[:cf.numel()].cpu().numpy(), cf.cpu().numpy(), equal_nan=True)
    assert np.array_equal(mm[:mf.numel()].cpu().numpy(), mf.cpu().numpy(), equal_nan=True)
    assert torch.equal(sm[:few.size], sf)
    assert int(sf[1]) & apm.ST_PIVOT_CORRECTED and int(sf[3]) & apm.ST_NONFINITE_INPUT
    c0 = apm.cdet_connected_varlen(A, ao[:few.size].contiguous(), nt[:few.size].contiguous())
    assert np.array_equal(c0.cpu().numpy(), cf.cpu().numpy(), equal_nan=True)
    row = np.concatenate([[0], np.cumsum(1 << few.astype(np.int64))])
    for b in range(7):
        n = int(few[b])
        x = torch.as_tensor(flat[off[b]:off[b] + n * n].reshape(1, n, n)).cuda()
        c1 = apm.cdet_connected(x)[0]
        assert np.array_equal(cf[row[b]:row[b + 1]].cpu().numpy(), c1.cpu().numpy(), equal_nan=True), b
    apm.tune_options_set(0, 1, 0)                       # fewer slots than these items' weights take
    try:
        c2 = apm.cdet_connected_varlen(A, ao[:few.size].contiguous(), nt[:few.size].contiguous())
    finally:
        apm.tune_options_set(0, 0, 0)
    assert np.array_equal(c2.cpu().numpy(), cf.cpu().numpy(), equal_nan=True)


# orders 11 and 12: clusters of 8, 4 and 2 CTAs per matrix, and one CTA each
@pytest.mark.parametrize("n,batch", [(11, 32), (11, 76), (11, 77), (12, 10), (12, 32), (12, 76), (12, 77)])
def test_clusters(apm, n, batch):
    d = torch.as_tensor(mixed(n, batch, 9000 + n)).cuda()
    e = torch.as_tensor(mixed(n, batch, 9100 + n)).cuda()
    many = torch.arange(200).cuda() % batch          # the same matrices in a call of one CTA each
    for f in (lambda x, y: apm.cdet_connected(x, return_minors=True, return_status=True),
              lambda x, y: apm.cdet_connected(x, y, return_minors=True, return_status=True),
              lambda x, y: apm.cdet_connected(x, single_det=True, return_status=True, piv_threshold=0.5),
              lambda x, y: (apm.cdet_from_weights(apm.cdet_connected(x, single_det=True)),)):
        rows_equal(f(d[many], e[many]), f(d, e), list(range(batch)))
