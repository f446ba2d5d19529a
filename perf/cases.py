"""What a user of the library has it compute: the cases its speed is measured on.

Every case is one call of a public entry point (``apm``, ``mc``) on matrices of the
kind the method meets: Green's functions of Monte Carlo vertex configurations
(``inputs``), at the orders and batch sizes of the repository's own workloads, from
one configuration to the 65536 of the benchmark, with odd sizes between.
"""
import functools
import math

import numpy as np
import torch

from paper_2104_07638_gb300 import apm, inputs, mc


def listed():
    return [
        # one configuration, every subset: the first thing a user tries, and a single chain's step
        {"name": "cdet_one_n10", "op": "cdet", "n": 10, "batch": 1, "kind": "gauss", "minors": True, "spins": False,
         "single": False},
        # the high orders of a series run on few configurations: each is costly
        {"name": "cdet_few_n14", "op": "cdet", "n": 14, "batch": 24, "kind": "hubbard", "minors": False,
         "spins": False, "single": False},
        # spin-polarised weights (two different matrices), minors and status read back, a ragged batch
        {"name": "cdet_spins_n9", "op": "cdet", "n": 9, "batch": 777, "kind": "hubbard", "minors": True,
         "spins": True, "single": False},
        # the benchmark's batch: minors and connected sums of 65536 configurations of order 12
        {"name": "cdet_batch_n12", "op": "cdet", "n": 12, "batch": 65536, "kind": "hubbard", "minors": True,
         "spins": False, "single": False},
        # one Metropolis step of 16384 walkers at a low order, where a series spends most of its samples
        {"name": "mc_step_n6", "op": "mc", "n": 6, "batch": 16384, "learned": False},
        # a batch of walkers of all orders in one call
        {"name": "uneven_4to16", "op": "uneven", "lo": 4, "hi": 16, "batch": 16384, "minors": True},
        # all minors without the recursion, a few matrices of high order
        {"name": "minors_n16", "op": "minors", "n": 16, "batch": 40},
        # real-time sums with their lower orders, one per walker
        {"name": "keldysh_n9", "op": "keldysh", "n": 9, "batch": 1000, "partial": True},
        # both spins under one shared Keldysh assignment, a small set of walkers
        {"name": "keldysh2_n8", "op": "keldysh2", "n": 8, "batch": 300, "partial": False},
        # bosonic weights: permanents of all subsets
        {"name": "perm_n12", "op": "perm", "n": 12, "batch": 512},
        # expansion around a superconducting state: block minors and their connected sums
        {"name": "nambu_n8", "op": "nambu", "n": 8, "batch": 2048},
        # two vertex types per vertex, summed over the types
        {"name": "two_type_n7", "op": "two_type", "n": 7, "batch": 3000},
    ]


# family: smallest and largest order, largest batch
_RANGES = {"cdet": (3, 16, 65536), "mc": (3, 12, 16384), "uneven": (4, 16, 8192), "minors": (4, 22, 65536),
           "keldysh": (2, 12, 65536), "keldysh2": (2, 10, 32768), "perm": (3, 14, 32768), "nambu": (2, 13, 65536),
           "two_type": (2, 10, 32768)}
_MOST = {"flops": 2.0e10, "bytes": 2.5e9}


def draw(rng):
    op = rng.choice(["cdet", "cdet", "cdet", "mc", "uneven", "minors", "keldysh", "keldysh2", "perm", "nambu",
                     "two_type"])
    lo, hi, most = _RANGES[op]
    n = rng.randint(lo, hi)
    case = {"op": op, "n": n}
    if op == "cdet":
        spins = rng.random() < 0.25
        case.update(kind=rng.choice(["hubbard", "hubbard", "gauss"]), minors=rng.random() < 0.5, spins=spins,
                    single=not spins and rng.random() < 0.2)
    elif op == "uneven":
        del case["n"]
        a, b = sorted((rng.randint(lo, hi), rng.randint(lo, hi)))
        case.update(lo=a, hi=b, minors=rng.random() < 0.5)
    elif op == "mc":
        case.update(learned=rng.random() < 0.5)          # moves filtered by the surrogate network first
    elif op in ("keldysh", "keldysh2"):
        case.update(partial=rng.random() < 0.5)
    one = work(dict(case, batch=1))
    cap = min(most, int(_MOST["flops"] / one["flops"]), int(_MOST["bytes"] / one["bytes"]))
    least = 64 if op in ("mc", "uneven") else 1
    cap = max(cap, least)
    case["batch"] = int(round(math.exp(rng.uniform(math.log(least), math.log(cap)))))
    return case


# --- inputs -------------------------------------------------------------------


def _gpu(x):
    return torch.as_tensor(x).cuda()


def _matrices(kind, n, batch, seed):
    make = inputs.gaussian_plus_2I if kind == "gauss" else inputs.hubbard_batch
    return make(n, batch, seed) if kind == "gauss" else make(batch, n, seed)


_tables = {}


def _nambu(batch, n, seed):
    if "nambu" not in _tables:
        _tables["nambu"] = inputs.nambu_g0_table()
    x, y, m = inputs.hubbard_vertices(batch, n, seed, mtau=inputs.NAMBU_MTAU)
    dx = np.abs(x[:, :, None] - x[:, None, :])
    dy = np.abs(y[:, :, None] - y[:, None, :])
    dt = m[:, :, None] - m[:, None, :] + (inputs.NAMBU_MTAU - 1)
    blocks = _tables["nambu"][dx, dy, dt]
    return np.ascontiguousarray(blocks.transpose(0, 1, 3, 2, 4).reshape(batch, 2 * n, 2 * n))


def _orders(case):
    return inputs.varlen_orders(case["batch"], case["lo"], case["hi"])


def _mats(case, seed):
    """The matrices of a case, on the host."""
    op, b, n = case["op"], case["batch"], case.get("n")
    if op == "cdet":
        up = _matrices(case["kind"], n, b, seed)
        return (up, _matrices(case["kind"], n, b, seed + 7919)) if case["spins"] else (up,)
    if op == "uneven":
        return inputs.hubbard_varlen(_orders(case), seed=seed)
    if op == "minors":
        return (inputs.hubbard_batch(b, n, seed),)
    if op == "keldysh":
        return (inputs.keldysh_batch(b, n, seed),)
    if op == "keldysh2":
        return inputs.keldysh2_batch(b, n, seed)
    if op == "perm":
        return (inputs.perm_batch(n, b, seed),)
    if op == "nambu":
        return (_nambu(b, n, seed),)
    return (inputs.two_type_batch(b, n, seed),)


def prepare(case, seed):
    case = dict(case)
    if case["op"] == "mc":
        if "g0" not in _tables:
            _tables["g0"] = _gpu(inputs.hubbard_g0_table())
        w = mc.Walkers(case["batch"], case["n"], _tables["g0"], inputs.HUB_WIN, inputs.HUB_MTAU, seed=seed)
        state = {"case": case, "walkers": w}
        if case["learned"]:
            state["net"] = mc.Surrogate(seed=seed, max_batch=case["batch"])
            w.init_surrogate(state["net"])
        return state
    state = {"case": case, "mats": [_gpu(x) for x in _mats(case, seed)]}
    if case["op"] == "uneven":
        state["n"] = _gpu(_orders(case))
        state["c_off"] = apm.varlen_out_offsets(state["n"])
    return state


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "mc":
        w = state["walkers"]
        if case["learned"]:
            w.step_da(state["net"])
            return w.X, w.weight, w.sign, w.s_cur
        w.step_plain()
        return w.X, w.weight, w.sign, w.c
    mats = state["mats"]
    if op == "cdet":
        return apm.cdet_connected(mats[0], mats[1] if case["spins"] else None, single_det=case["single"],
                                  return_minors=case["minors"], return_status=case["spins"])
    if op == "uneven":
        return apm.cdet_connected_varlen(mats[0], mats[1], state["n"], n_max=case["hi"], c_off=state["c_off"],
                                         return_minors=case["minors"])
    if op == "minors":
        return apm.all_minors(mats[0])
    if op == "keldysh":
        return apm.keldysh_sum(mats[0], partial=case["partial"], return_status=True)
    if op == "keldysh2":
        return apm.keldysh2_sum(mats[0], mats[1], partial=case["partial"], return_status=True)
    if op == "perm":
        return apm.perm_minors(mats[0])
    if op == "nambu":
        return apm.nambu_cdet(mats[0], return_minors=True, return_status=True)
    return apm.two_type_cdet(mats[0], return_weights=True, return_status=True)


# --- the work of one pass -----------------------------------------------------


def _tree(n):
    return 2 * sum(2 ** l * (n - l - 1) ** 2 for l in range(n)) + 2 * (2 ** n - 1)


def _recursion(n):
    """Eq. recursion, or the fast subset convolution where that is the shorter (two ranked
    transforms and a logarithm: about n^2 2^n (1 + 1/3))."""
    return min((3 ** n - 1) - (2 ** n - 1), 4 * n * n * 2 ** n // 3)


def _keldysh(n):
    return 8 * sum(2 ** (l + 1) * 2 * (n - l - 1) * (2 * (n - l - 1) - 1) for l in range(n)) + 26 * 2 ** n


def _xnor(n):
    return sum(2 ** l * (16 * (n - l - 1) ** 2 + 12 * (n - l - 1) + 9) for l in range(n))


def _nand(n):
    return sum(3 ** l * 2 * (8 * (n - l - 1) ** 2 - 2 * (n - l - 1) + 3) for l in range(n))


def work(case):
    op, b, n = case["op"], case["batch"], case.get("n")
    if op == "uneven":
        k = range(case["lo"], case["hi"] + 1)
        rows = 2 if case["minors"] else 1
        return {"bytes": b * sum(8 * m * m + 8 * rows * 2 ** m + 20 for m in k) / len(k),
                "flops": b * sum(_tree(m) + _recursion(m) + 2 ** m for m in k) / len(k)}
    N = 2 ** n
    if op == "cdet":
        mats = 2 if case["spins"] else 1
        return {"bytes": b * (8 * mats * n * n + 8 * N * (1 + (mats if case["minors"] else 0))),
                "flops": b * (mats * _tree(n) + _recursion(n) + N)}
    if op == "mc":
        return {"bytes": b * (24 * n + 40 + 8 * N), "flops": b * (_tree(n) + _recursion(n) + N)}
    if op == "minors":
        return {"bytes": b * (8 * n * n + 8 * N), "flops": b * _tree(n)}
    if op == "keldysh":
        return {"bytes": b * (64 * n * n + 16 + (16 * (n + 1) if case["partial"] else 0)), "flops": b * _keldysh(n)}
    if op == "keldysh2":
        return {"bytes": b * (128 * n * n + 16 + (16 * (n + 1) if case["partial"] else 0)),
                "flops": 2 * b * _keldysh(n) + 20 * b * N}
    if op == "perm":
        return {"bytes": b * (8 * n * n + 8 * N), "flops": b * (2 * 3 ** n + n * N)}
    if op == "nambu":
        return {"bytes": b * (32 * n * n + 16 * N), "flops": b * (_xnor(n) + _recursion(n))}
    return {"bytes": b * (32 * n * n + 16 * N), "flops": b * (_nand(n) + _recursion(n))}


# --- the same in plain torch, 64 bits -------------------------------------------


def _bits(S, n):
    return [i for i in range(n) if S >> i & 1]


def _dets(A, rows):
    """det of the kept rows and columns of every matrix; 1 where none is kept."""
    if not rows:
        return torch.ones(A.shape[0], dtype=A.dtype, device=A.device)
    i = torch.tensor(rows, device=A.device)
    return torch.linalg.det(A[:, i][:, :, i])


def _exact_minors(A):
    """All principal minors: each by its own pivoted elimination where there are few, else by
    Schur complements (element 0 first), the pivots of these matrices being well away from 0."""
    b, n, _ = A.shape
    if n <= 10 and b <= 4096:
        return torch.stack([_dets(A, _bits(S, n)) for S in range(1 << n)], 1)
    out = torch.ones((b, 1), dtype=A.dtype, device=A.device)
    W = A[:, None]                                       # (b, 2^l nodes, n-l, n-l)
    for _ in range(n):
        p = W[:, :, :1, :1]
        low = W[:, :, 1:, 1:]
        out = torch.cat([out, out * p[:, :, 0, 0]], 1)
        W = torch.cat([low, low - W[:, :, 1:, :1] * W[:, :, :1, 1:] / p], 1)
    return out


@functools.lru_cache(maxsize=1)
def _terms(n):
    """Per layer |S| = k of Eq. recursion: the sets S, and for each its proper subsets T that
    hold its lowest element."""
    masks = torch.arange(1 << n, device="cuda")
    pop = sum((masks >> i) & 1 for i in range(n))
    layers = []
    for k in range(1, n + 1):
        S = masks[pop == k]
        at = ((S[:, None] >> torch.arange(n, device="cuda")) & 1).nonzero()[:, 1].reshape(-1, k)
        U = torch.arange((1 << (k - 1)) - 1, device="cuda")
        T = (1 << at[:, :1]).expand(-1, U.numel()).to(torch.int32).clone()
        for i in range(k - 1):
            T += (((U >> i) & 1)[None] << at[:, i + 1:i + 2]).to(torch.int32)
        layers.append((S, T))
    return layers


def _exact_connected(a):
    """c[S] = a[S] - sum over the proper subsets T of S that hold its lowest element of c[T] a[S \\ T]."""
    b, N = a.shape
    c = torch.zeros_like(a)
    for S, T in _terms(N.bit_length() - 1):
        step = max(1, int(2.5e8 / (b * max(1, T.shape[1]))))
        for i in range(0, S.numel(), step):
            s, t = S[i:i + step], T[i:i + step].long()
            c[:, s] = a[:, s] - (c[:, t] * a[:, s[:, None] - t]).sum(-1)
    return c


def _connected(up, dn, single):
    mu = _exact_minors(up)
    md = mu if dn is None else _exact_minors(dn)
    c = _exact_connected(mu if single else mu * md)
    return c, mu if dn is None else torch.stack([mu, md], 1)


def _exact_permanents(A):
    b, n, _ = A.shape
    out = torch.zeros((b, 1 << n), dtype=A.dtype, device=A.device)
    masks = torch.arange(1 << n, device=A.device)
    r = torch.zeros((b, n, 1), dtype=A.dtype, device=A.device)       # row sums over the columns T
    for j in range(n):
        r = torch.cat([r, r + A[:, :, j:j + 1]], 2)
    size = sum((masks >> i) & 1 for i in range(n))
    sign = (1 - 2 * (size & 1)).to(A.dtype)
    for T in range(1 << n):
        p = torch.ones((b, 1), dtype=A.dtype, device=A.device)
        for i in range(n):
            q = p * r[:, i, T:T + 1]
            p = torch.cat([q * 0 if T >> i & 1 else p, q], 1)
        out += p * (1 - 2 * (bin(T).count("1") & 1))
    return out * sign


def _exact_keldysh(mats, n):
    """The sums over the assignments of the first d vertices, d = 0..n."""
    parts = []
    for d in range(n + 1):
        tot = 0
        for S in range(1 << d):
            rows = [2 * i + (S >> i & 1) for i in range(d)]
            v = 1
            for M in mats:
                v = v * _dets(M, rows)
            tot = tot + v
        parts.append(tot)
    return torch.stack(parts, 1)


def exact(case, seed):
    op, b, n = case["op"], case["batch"], case.get("n")
    if op == "mc":
        return None                                      # its random numbers are the chain's own
    mats = [_gpu(x) for x in _mats(case, seed)]
    if op == "cdet":
        if b * 3 ** n > 1e11:
            return None
        parts = [_connected(mats[0][i:i + 8192], mats[1][i:i + 8192] if case["spins"] else None, case["single"])
                 for i in range(0, b, 8192)]
        c, m = (torch.cat(x) for x in zip(*parts))
        out = [c] + ([m] if case["minors"] else []) + ([None] if case["spins"] else [])
        return out[0] if len(out) == 1 else tuple(out)
    if op == "uneven":
        orders, (flat, off) = _orders(case), mats
        row = np.concatenate([[0], np.cumsum(1 << orders.astype(np.int64))])
        c = torch.zeros(int(row[-1]), dtype=torch.float64, device="cuda")
        m = torch.zeros_like(c)
        for k in np.unique(orders):
            sel = np.nonzero(orders == k)[0]
            A = flat[off[_gpu(sel)][:, None] + torch.arange(k * k, device="cuda")].reshape(-1, k, k)
            at = _gpu(row[sel])[:, None] + torch.arange(1 << k, device="cuda")
            c[at], m[at] = _connected(A, None, False)
        return (c, m) if case["minors"] else c
    if op == "minors":
        return torch.cat([_exact_minors(mats[0][i:i + 4096]) for i in range(0, b, 4096)]) if b << n <= 1 << 28 else None
    if op in ("keldysh", "keldysh2"):
        if n > 11 or b << n > 1 << 23:
            return None
        p = _exact_keldysh(mats, n)
        return (p[:, n], p, None) if case["partial"] else (p[:, n], None)
    if op == "perm":
        return _exact_permanents(mats[0]) if n <= 12 and b << n <= 1 << 24 else None
    if op == "nambu":
        if n > 11 or b << n > 1 << 23:
            return None
        a = torch.stack([_dets(mats[0], [2 * i + s for i in _bits(S, n) for s in (0, 1)]) for S in range(1 << n)], 1)
        return _exact_connected(a), a, None
    if n > 8 or b * 3 ** n > 1 << 24:
        return None
    a = torch.zeros((b, 1 << n), dtype=torch.float64, device="cuda")
    for t in range(3 ** n):
        digits = [t // 3 ** i % 3 for i in range(n)]
        a[:, sum(1 << i for i in range(n) if digits[i])] += _dets(mats[0], [2 * i + d - 1 for i, d in enumerate(digits) if d])
    return _exact_connected(a), a, None
