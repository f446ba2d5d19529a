"""What the choice of a route must not change: status words, the possibility of
capture, scratch that serves every smaller batch, results."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
from paper_2104_07638_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def apm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_07638_gb300 import apm as m
    m.lib()
    m.tune_set(None)
    m.tune_options_set(0, 0, 0)
    return m


def zero_pivot_at(n, kept, e, rng):
    """A matrix whose pivot of element e is zero where exactly the set `kept` of the
    elements below e is kept, and about 2 elsewhere."""
    A = 2.0 * np.eye(n) + 0.2 * rng.standard_normal((n, n))
    k = [i for i in range(e) if kept >> i & 1]
    A[e, e] = A[e, k] @ np.linalg.solve(A[np.ix_(k, k)], A[k, e]) if k else 0.0
    return A


# a pivot corrected in the subtree of one CTA of the cluster only: its status bit
# reaches the status word whichever CTA that is, with one matrix and with two
@pytest.mark.parametrize("n,batch", [(11, 32), (12, 10), (12, 40)])
def test_cluster_status(apm, n, batch):
    rng = np.random.default_rng(9200 + n)
    A = np.stack([zero_pivot_at(n, b % 8, 5 + b % 3, rng) for b in range(batch)])
    A[8] = I.gaussian_plus_2I(n, 1, seed=3)[0]
    A[9, n - 1, 0] = np.nan
    B = np.stack([zero_pivot_at(n, (3 * b + 1) % 8, 6, rng) if b % 2 else I.gaussian_plus_2I(n, 1, seed=b)[0]
                  for b in range(batch)])
    d, e = torch.as_tensor(A).cuda(), torch.as_tensor(B).cuda()
    many = torch.arange(200).cuda() % batch          # the same matrices in a call of one CTA each
    for x, y in ((d, None), (d, e), (e, d)):
        ref = apm.cdet_connected(x[many], None if y is None else y[many], return_minors=True, return_status=True)
        assert int(ref[2][0]) & apm.ST_PIVOT_CORRECTED
        for _ in range(20):
            got = apm.cdet_connected(x, y, return_minors=True, return_status=True)
            for g, r in zip(got, ref):
                assert np.array_equal(g.cpu().numpy(), r[:batch].cpu().numpy(), equal_nan=True)


CAPTURE = """
import ctypes, torch
from paper_2104_07638_gb300 import apm
g = torch.Generator(device='cuda').manual_seed(1)
def mats(b, n):
    return torch.eye(n, device='cuda', dtype=torch.float64) + \
        0.1 * torch.randn((b, n, n), generator=g, device='cuda', dtype=torch.float64)
apm.cdet_connected(mats(30000, 6))              # lane groups
torch.cuda.synchronize()
s = ctypes.c_void_p()
assert ctypes.CDLL('libcuda.so.1').cuStreamCreate(ctypes.byref(s), 0) == 0
for n, b in ((10, 3), (12, 100), (14, 3)):
    A = mats(b, n)
    torch.cuda.synchronize()
    G = torch.cuda.CUDAGraph()
    with torch.cuda.graph(G, stream=torch.cuda.ExternalStream(s.value)):
        c = apm.cdet_connected(A)
    G.replay()
    torch.cuda.synchronize()
    assert torch.equal(c, apm.cdet_connected(A))
print('captured')
"""


def test_capture_after_a_first_call_by_lane_groups(apm):
    """Any first call uploads the constant tables: the calls after it can be
    captured, on a stream that waits for the legacy one too."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CAPTURE], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured" in r.stdout, r.stderr[-2000:]


# uneven batches without orders above 11, on both sides of every change of the
# CTA's width, one matrix and two per item, against fixed-order calls; few and many
# of the largest order where that decides
@pytest.mark.parametrize("lo,hi,batch", [(1, 3, 50), (1, 6, 500), (1, 8, 456), (1, 8, 457), (1, 9, 456), (1, 9, 457),
                                         (9, 9, 361), (9, 9, 500), (1, 9, 1100), (1, 9, 1101), (9, 10, 1000),
                                         (1, 10, 2000), (1, 10, 2001), (11, 11, 457), (11, 11, 1000), (10, 11, 1500),
                                         (1, 11, 3100), (1, 11, 3101)])
def test_uneven_small_orders(apm, lo, hi, batch):
    rng = np.random.default_rng(9300 + hi)
    orders = rng.integers(lo, hi + 1, batch).astype(np.int32)
    orders[:3] = hi
    off = np.concatenate([[0], np.cumsum(orders.astype(np.int64) ** 2)])[:-1]
    flat = rng.standard_normal((2, int((orders.astype(np.int64) ** 2).sum())))
    flat[0, off[1]:off[1] + hi * hi] = 0.0                 # corrected at every pivot
    flat[0, off[2]] = np.inf
    A, B = (torch.as_tensor(x).cuda() for x in flat)
    ao, nt = torch.as_tensor(off).cuda(), torch.as_tensor(orders).cuda()
    co = apm.varlen_out_offsets(nt)
    for dn in (None, B):
        mats = 1 if dn is None else 2
        c, mo, st = apm.cdet_connected_varlen(A, ao, nt, A_dn=dn, return_minors=True, return_status=True)
        for m in range(1, hi + 1):
            at = torch.as_tensor(np.nonzero(orders == m)[0]).cuda()
            if at.numel() == 0:
                continue
            sq = torch.arange(m * m, device="cuda")
            x = A[ao[at][:, None] + sq].reshape(-1, m, m)
            y = None if dn is None else B[ao[at][:, None] + sq].reshape(-1, m, m)
            cr, mr, sr = apm.cdet_connected(x, y, return_minors=True, return_status=True)
            S = torch.arange(1 << m, device="cuda")
            got = c[co[at][:, None] + S]
            assert np.array_equal(got.cpu().numpy(), cr.cpu().numpy(), equal_nan=True), m
            S = torch.arange(mats << m, device="cuda")
            got = mo[mats * co[at][:, None] + S].reshape(mr.shape)
            assert np.array_equal(got.cpu().numpy(), mr.cpu().numpy(), equal_nan=True), m
            assert torch.equal(st[at], sr), m


# XNOR minors: whole matrices from where halves would take a second round
@pytest.mark.parametrize("n,batch", [(10, 760), (10, 761), (11, 911), (11, 912), (12, 1216)])
def test_xnor_whole_from(apm, n, batch):
    d = torch.as_tensor(I.nambu_batch(64, n, seed=9400 + n)).cuda()
    few = apm.xnor_minors(d, return_status=True)
    at = torch.arange(batch).cuda() % 64
    big = apm.xnor_minors(d[at], return_status=True)
    for g, r in zip(big, few):
        assert torch.equal(g, r[at])
    sizes = [apm.workspace_size(apm.OP_XNOR_MINORS, n, b) for b in (1, 200, 456, 760, 761, 911, 912, 1520, 3000)]
    assert sizes == sorted(sizes)


# Keldysh sums of batches above one round of warps: whole where splitting gains no
# round (then also bit for bit the same matrices of the uneven batch), else split;
# against a batch of one (other chunks: a rounding apart)
@pytest.mark.parametrize("n,batch,whole", [(10, 2736, False), (10, 3648, True), (11, 3300, True), (12, 1900, False)])
def test_keldysh_rounds(apm, n, batch, whole):
    d = torch.as_tensor(I.keldysh_batch(32, n, seed=9500 + n)).cuda()
    at = torch.arange(batch).cuda() % 32
    s, p = apm.keldysh_sum(d[at], partial=True)
    assert torch.equal(s, s[at]) and torch.equal(p, p[at])
    o = torch.arange(32).cuda() * (4 * n * n)
    u = apm.keldysh_sum_varlen(d.reshape(-1), o, torch.full((32,), n, dtype=torch.int32, device="cuda"))
    if whole:
        assert torch.equal(s[:32], u)
    scale = torch.as_tensor(oracle.keldysh_scale(d.cpu().numpy())).cuda()
    one = apm.keldysh_sum(d[:1])
    assert bool((abs(s[:32] - u) <= 1e-10 * scale).all()) and bool((abs(s[:1] - one) <= 1e-10 * scale[:1]).all())


@pytest.mark.parametrize("n,batch", [(8, 3000), (8, 3648), (9, 5472)])
def test_keldysh2_rounds(apm, n, batch):
    u, d = (torch.as_tensor(x).cuda() for x in I.keldysh2_batch(32, n, seed=9600 + n))
    at = torch.arange(batch).cuda() % 32
    s, p = apm.keldysh2_sum(u[at], d[at], partial=True)
    w, q = apm.keldysh2_sum(u[at[:1824]], d[at[:1824]], partial=True)    # one round of whole pairs
    assert torch.equal(s[:1824], w) and torch.equal(p[:1824], q) and torch.equal(s, s[at])


# scratch sized for a batch serves every smaller one, split into more chunks or not
@pytest.mark.parametrize("n", [9, 10, 11, 12, 14])
def test_keldysh_scratch_serves_smaller_batches(apm, n):
    bs = sorted({1, 2, 3, 57, 228, 300, 456, 500, 911, 912, 913, 1000, 1824, 1825, 2052, 3648, 7296, 14592, 14593,
                 40000} | set(range(1, 4000, 61)))
    sizes = [apm.workspace_size(apm.OP_KELDYSH, n, b) for b in bs]
    assert sizes == sorted(sizes)
    M = torch.as_tensor(I.keldysh_batch(300, n, seed=9700 + n)).cuda()
    nb = apm.workspace_size(apm.OP_KELDYSH, n, 500)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    for b in (1, 57, 300):
        s = torch.empty((b, 2), dtype=torch.float64, device="cuda")
        apm._check(apm.lib().apm_keldysh_sum(apm._ptr(M), n, b, 0, apm._ptr(s), None, None, apm._ptr(ws), nb,
                                             apm._stream(M)), "apm_keldysh_sum")
        assert torch.equal(torch.view_as_complex(s), apm.keldysh_sum(M[:b]))


# scratch of a few two-spin pairs: stacks for the warps they can occupy, no more,
# and one that serves every smaller batch
@pytest.mark.parametrize("n,most", [(8, 0.2e6), (10, 0.8e6), (12, 4.2e6), (14, 27e6), (16, 155e6)])
def test_keldysh2_scratch(apm, n, most):
    assert apm.workspace_size(apm.OP_KELDYSH2, n, 1) <= most
    bs = sorted({1, 2, 7, 28, 57, 300, 1824, 1825, 3648, 14592, 14593, 40000} | set(range(1, 4000, 61)))
    sizes = [apm.workspace_size(apm.OP_KELDYSH2, n, b) for b in bs]
    assert sizes == sorted(sizes)
    if n > 10:
        return
    u, d = (torch.as_tensor(x).cuda() for x in I.keldysh2_batch(300, n, seed=9800 + n))
    nb = apm.workspace_size(apm.OP_KELDYSH2, n, 500)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    for b in (1, 57, 300):
        s = torch.empty((b, 2), dtype=torch.float64, device="cuda")
        apm._check(apm.lib().apm_keldysh2_sum(apm._ptr(u), apm._ptr(d), n, b, 0, apm._ptr(s), None, None, apm._ptr(ws),
                                              nb, apm._stream(u)), "apm_keldysh2_sum")
        assert torch.equal(torch.view_as_complex(s), apm.keldysh2_sum(u[:b], d[:b]))


# scratch of an uneven batch: rows of terms for the items there are, not 64 MB for
# any two, and enough for every smaller batch
@pytest.mark.parametrize("n_max", [13, 14, 15, 16])
def test_uneven_scratch(apm, n_max):
    slots = 456 * (3 << n_max) * 8                       # three CTAs per SM
    most = {13: 9, 14: 28, 15: 75, 16: 75}[n_max] * 8192     # bytes of rows per item
    for b in (1, 2, 4):
        size = apm.workspace_size(apm.OP_CDET_VARLEN, n_max, b)
        assert slots <= size <= slots + b * most + 1024
    bs = sorted({1, 2, 8, 100, 109, 110, 292, 293, 910, 911, 1024, 1025, 5000, 70000} | set(range(1, 1200, 37)))
    sizes = [apm.workspace_size(apm.OP_CDET_VARLEN, n_max, b) for b in bs]
    assert sizes == sorted(sizes)


# the CTA's width at orders 10 and 11, one matrix and two
@pytest.mark.parametrize("n,batch", [(10, 1520), (10, 1521), (11, 608), (11, 609), (11, 912), (11, 913), (11, 1216),
                                     (11, 1217), (11, 1368), (11, 1369)])
def test_cta_widths(apm, n, batch):
    few = 200                                        # one round of wide CTAs
    A = torch.as_tensor(I.gaussian_plus_2I(n, few, seed=n)).cuda()
    B = torch.as_tensor(I.hubbard_batch(few, n, seed=n)).cuda()
    at = torch.arange(batch).cuda() % few
    for y in (None, A):
        ref = apm.cdet_connected(B, y, return_minors=True, return_status=True)
        got = apm.cdet_connected(B[at], None if y is None else y[at], return_minors=True, return_status=True)
        for g, r in zip(got, ref):
            assert torch.equal(g, r[at])


# both sides of the lines between CTAs and lane groups
@pytest.mark.parametrize("n,lines", [(4, (457, 1900)), (5, (1800, 2000, 2200)), (6, (2000, 2200, 11500)),
                                     (7, (5000, 5600, 20000)), (8, (10500, 22000))])
def test_lane_group_lines(apm, n, lines):
    A = torch.as_tensor(I.gaussian_plus_2I(n, 64, seed=40 + n)).cuda()
    A[3] = 0.0
    A[5, 0, 1] = float("nan")
    c, m, st = (x.nan_to_num(nan=1.5e300) if x.is_floating_point() else x
                for x in apm.cdet_connected(A, return_minors=True, return_status=True))
    w = apm.all_minors(A[6:])
    cw = apm.cdet_from_weights(w)
    for b in (x + y for x in lines for y in (-1, 0)):
        at = torch.arange(b).cuda() % 64
        got = apm.cdet_connected(A[at], return_minors=True, return_status=True)
        for g, r in zip(got, (c, m, st)):
            assert torch.equal(g.nan_to_num(nan=1.5e300) if g.is_floating_point() else g, r[at])
        assert torch.equal(apm.all_minors(A[at]).nan_to_num(nan=1.5e300), m[at])
        at = torch.arange(b).cuda() % 58
        assert torch.equal(apm.cdet_from_weights(w[at]), cw[at])


# uneven batches of orders 13..15 by blocks on many CTAs or, where that would take
# longer, with one CTA per matrix: fixed-order results either way, flagged matrices
# among them
@pytest.mark.parametrize("orders", [[13] * 300, [13] * 100, [13, 14] * 430, [12, 13, 14] * 90, [14] * 460, [15, 13] * 20])
def test_uneven_blocks_or_not(apm, orders):
    uniq, o = 16, np.asarray(orders, dtype=np.int32)
    mats = {m: I.hubbard_batch(uniq, m, seed=9900 + m) for m in set(orders)}
    for m in mats:
        mats[m][3] = 0.0                                   # corrected at every pivot
        mats[m][5, 0, m - 1] = np.nan
    flat = np.concatenate([mats[m][b % uniq].ravel() for b, m in enumerate(orders)])
    off = np.concatenate([[0], np.cumsum(o.astype(np.int64) ** 2)])[:-1]
    A, ao, nt = (torch.as_tensor(x).cuda() for x in (flat, off, o))
    c, mo, st = apm.cdet_connected_varlen(A, ao, nt, return_minors=True, return_status=True)
    co = apm.varlen_out_offsets(nt)
    for m in mats:
        ref = apm.cdet_connected(torch.as_tensor(mats[m]).cuda(), return_minors=True, return_status=True)
        at = np.nonzero(o == m)[0]
        for x, r in ((c, ref[0]), (mo, ref[1])):
            for lo in range(0, at.size, 64):               # (bits, so that NaN equals itself)
                k = torch.as_tensor(at[lo:lo + 64]).cuda()
                got = x[co[k][:, None] + torch.arange(1 << m, device="cuda")]
                assert torch.equal(got.nan_to_num(nan=1.5e300), r[k % uniq].nan_to_num(nan=1.5e300)), m
        k = torch.as_tensor(at).cuda()
        assert torch.equal(st[k], ref[2][k % uniq])


# the fast subset convolution: a last round by tiles up to where a whole one is faster
@pytest.mark.parametrize("n,batch", [(12, 64), (12, 65), (13, 440), (13, 441), (14, 450), (14, 451), (13, 456 + 441)])
def test_fsc_last_round(apm, n, batch):
    w = torch.rand((32, 1 << n), dtype=torch.float64, device="cuda",
                   generator=torch.Generator(device="cuda").manual_seed(n))
    at = torch.arange(batch).cuda() % 32
    assert torch.equal(apm.cdet_from_weights_fsc(w[at]), apm.cdet_from_weights_fsc(w)[at])


# installed lane-group tables reach the lane groups too, where most of a group's
# partial sums are one lane's: the largest groups, next to none, some layers, against
# the one-CTA-per-matrix kernel under the same table
@pytest.mark.parametrize("n,batch", [(4, 3000), (5, 1800), (5, 40000), (6, 3600), (6, 40000), (7, 6000), (7, 30000),
                                     (8, 22000)])
def test_lane_groups_under_installed_tables(apm, n, batch):
    A = torch.as_tensor(I.gaussian_plus_2I(n, 200, seed=60 + n)).cuda()
    at = torch.arange(batch).cuda() % 200
    tables = [[min(5, k - 1) if 2 <= k <= n else 0 for k in range(17)], [int(k == n) for k in range(17)],
              [k % 2 if 2 <= k <= n else 0 for k in range(17)], [min(2, k - 1) if 2 <= k <= n else 0 for k in range(17)]]
    try:
        for r in tables:
            packed = sum(x << (3 * k) for k, x in enumerate(r))
            apm.tune_set([packed if m == n else 0 for m in range(17)])
            few, big = apm.cdet_connected(A), apm.cdet_connected(A[at])
            assert torch.equal(big, few[at]), r
    finally:
        apm.tune_set(None)


def test_lane_groups_are_timed_on_the_uneven_kernel(apm, monkeypatch):
    """The tables serve the uneven batch: they are not chosen by fixed-order calls,
    which take other kernels at these orders."""
    from paper_2104_07638_gb300 import batch

    def fixed(*a, **k):
        raise AssertionError("a fixed-order call was timed")
    monkeypatch.setattr(apm, "cdet_connected", fixed)
    monkeypatch.setattr(batch, "_cache_path", lambda: str(batch._build.BUILD) + "/tune_test.json")
    try:
        tuned = batch.autotune(orders=(7, 8), fsc_orders=(), reps=5, use_cache=False, tune_launch=False)
        for n in (7, 8):
            t = tuned["timings"][f"lane_groups_n{n}"]
            assert t["tuned_ms"] <= t["default_ms"]
    finally:
        apm.tune_set(None)
        apm.tune_options_set(0, 0, 0)


# orders above 12 level by level or with one CTA per matrix, on both sides of each line
@pytest.mark.parametrize("n,batch", [(13, 235), (13, 236), (13, 304), (13, 305), (13, 360), (13, 361), (14, 275),
                                     (14, 276), (14, 406), (15, 288), (15, 305), (13, 456 + 300), (13, 456 + 400)])
def test_split_lines(apm, n, batch):
    A = I.hubbard_batch(16, n, seed=70 + n)
    A[3] = 0.0
    A[5, 0, n - 1] = np.inf
    d = torch.as_tensor(A).cuda()
    at = torch.arange(batch).cuda() % 16
    ref = apm.cdet_connected(d, return_status=True)
    got = apm.cdet_connected(d[at], return_status=True)
    assert torch.equal(got[1], ref[1][at])
    for lo in range(0, batch, 64):
        assert torch.equal(got[0][lo:lo + 64].nan_to_num(nan=1.5e300), ref[0][at[lo:lo + 64]].nan_to_num(nan=1.5e300))
