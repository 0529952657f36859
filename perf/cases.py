"""The calls that programs make of this package, as cases to time and compare.

A case is a dict of plain values. Its "kind" names the entry point:

  table      one table of a zero-mean state (fn, precision, M, kmax), into an
             output and a workspace that the program keeps;
  call       the same through the bare call, which allocates both and checks
             the status, as a small script does;
  displaced  one table of a displaced state, FP64;
  fit        one step of fitting squeezing and transmissions: the covariance
             model, its cumulant table, a weighted squared loss and the gradient;
  batch      the click-cumulant tables of n ragged instances in one launch;
  sample     n bitstrings drawn from a spin-cumulant table.

States are lossy squeezed-light interferometers (Haar unitary, xxpp, hbar = 2)
with the squeezing and loss ranges of the package's workloads.
"""
from __future__ import annotations

import math
from math import comb

import numpy as np
import torch

import paper_2511_14923_gb300 as gbs

TABLE_FNS = ("vacuum_probs", "click_moments", "cumulants", "spin_correlators", "spin_cumulants")


def listed():
    return [
        # a script that looks at one small state: launches and host work are all there is
        {"name": "call_m8_k3", "kind": "call", "fn": "cumulants", "precision": "fp64", "M": 8, "kmax": 3},
        # a mid-size state in a parameter scan, at the default precision
        {"name": "cumulants_m50_k4_fp64", "kind": "table", "fn": "cumulants", "precision": "fp64", "M": 50, "kmax": 4},
        # the order-5 table of an interferometer between the two sizes above and below, FP64 throughout
        {"name": "cumulants_m111_k5_fp64", "kind": "table", "fn": "cumulants", "precision": "fp64", "M": 111, "kmax": 5},
        # the headline table: 144 outputs, orders up to 5, refined FP32 determinants
        {"name": "cumulants_m144_k5_fp32r", "kind": "table", "fn": "cumulants", "precision": "fp32r", "M": 144, "kmax": 5},
        # vacuum probabilities alone (loss calibration), an odd size
        {"name": "vacuum_m77_k5_fp32r", "kind": "table", "fn": "vacuum_probs", "precision": "fp32r", "M": 77, "kmax": 5},
        # the K = 3 sampler's table for 144 outputs read through 8 time bins
        {"name": "spin_m1152_k3_fp64", "kind": "table", "fn": "spin_cumulants", "precision": "fp64", "M": 1152, "kmax": 3},
        # a state with coherent light in it
        {"name": "displaced_m97_k4", "kind": "displaced", "table": "kappa", "M": 97, "kmax": 4},
        # one fitting step, forward and backward
        {"name": "fit_m100_k4", "kind": "fit", "M": 100, "kmax": 4},
        # many small experiments of different sizes at once
        {"name": "batch_48", "kind": "batch", "precision": "fp32r", "n": 48, "M_lo": 16, "M_hi": 128},
        # drawing samples: the full emulator, the single-elision one at many modes, and the FP64 reference run
        {"name": "sample_k5_m144_fp32", "kind": "sample", "K": 5, "M": 144, "n": 8192, "batch": 8192, "precision": "fp32"},
        {"name": "sample_k3_m1152_fp32", "kind": "sample", "K": 3, "M": 1152, "n": 256, "batch": 256, "precision": "fp32"},
        {"name": "sample_k5_m100_fp64", "kind": "sample", "K": 5, "M": 100, "n": 256, "batch": 256, "precision": "fp64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["table"] * 5 + ["call", "displaced", "fit", "batch", "sample", "sample"])
    if kind in ("table", "call"):
        kmax = rng.choice([3, 4, 4, 5, 5]) if kind == "table" else rng.choice([2, 3, 4])
        lo, hi = {2: (8, 64), 3: (8, 1152), 4: (8, 300), 5: (16, 144)}[kmax]
        if kind == "call":
            hi = min(hi, 60)
        return {"kind": kind, "fn": rng.choice(("cumulants",) + TABLE_FNS), "precision": rng.choice(["fp64", "fp32r"]),
                "M": _log_int(rng, lo, hi), "kmax": kmax}
    if kind == "displaced":
        kmax = rng.choice([3, 4, 5])
        return {"kind": kind, "table": rng.choice(["p0", "mu", "kappa", "spin_kappa"]),
                "M": _log_int(rng, 12, {3: 300, 4: 144, 5: 100}[kmax]), "kmax": kmax}
    if kind == "fit":
        kmax = rng.choice([3, 4, 4, 5])
        return {"kind": kind, "M": _log_int(rng, 10, {3: 144, 4: 100, 5: 40}[kmax]), "kmax": kmax}
    if kind == "batch":
        lo = rng.randint(8, 32)
        return {"kind": kind, "precision": rng.choice(["fp32r", "fp32r", "fp64"]), "n": _log_int(rng, 4, 48), "M_lo": lo,
                "M_hi": rng.randint(lo + 8, 110)}
    K, precision = rng.choice([(3, "fp32"), (4, "fp32"), (5, "fp32"), (5, "fp32"), (3, "fp64"), (5, "fp64")])
    M = _log_int(rng, 16, {(3, "fp32"): 500, (3, "fp64"): 300, (5, "fp64"): 80}.get((K, precision), 144))
    batch = 128 * rng.randint(1, 2 if precision == "fp64" else 16)
    return {"kind": "sample", "K": K, "M": M, "n": max(1, batch - rng.randint(0, 120)), "batch": batch, "precision": precision}


# ---------------------------------------------------------------- inputs

def _state(M, rng, r_range=(0.8, 1.6), eta_range=(0.3, 0.5)):
    """U, r (squeezers on the first half of the modes) and eta of one interferometer."""
    z = rng.standard_normal((M, M)) + 1j * rng.standard_normal((M, M))
    q, rr = np.linalg.qr(z)
    d = np.diag(rr)
    r = np.zeros(M)
    r[: M // 2] = rng.uniform(*r_range, M // 2)
    return q * (d / np.abs(d))[None, :], r, rng.uniform(*eta_range, M)


def _covariance(U, r, eta):
    S = np.block([[U.real, -U.imag], [U.imag, U.real]])
    D = np.sqrt(np.concatenate([eta, eta]))
    V = D[:, None] * ((S * np.exp(np.concatenate([-2 * r, 2 * r]))[None, :]) @ S.T) * D[None, :] + np.diag(1 - D * D)
    return 0.5 * (V + V.T)


def _V(case, seed):
    """Covariance of a single-state case and (displaced) its first moments."""
    rng = np.random.default_rng([seed, case["M"], case.get("kmax", case.get("K"))])
    U, r, eta = _state(case["M"], rng)
    M = case["M"]
    alpha = 0.5 * (rng.standard_normal(M) + 1j * rng.standard_normal(M)) / np.sqrt(2.0)
    beta = np.sqrt(eta) * (U @ alpha)
    return _covariance(U, r, eta), np.concatenate([2 * beta.real, 2 * beta.imag])


def _fit_inputs(case, seed):
    """U, start (r, eta) and the covariance whose table is the target."""
    rng = np.random.default_rng([seed, case["M"], case["kmax"], 1])
    U, r, eta = _state(case["M"], rng, (0.5, 1.2), (0.3, 0.6))
    r2 = np.zeros_like(r)
    r2[: case["M"] // 2] = rng.uniform(0.5, 1.2, case["M"] // 2)
    return U, r, eta, _covariance(U, r2, rng.uniform(0.3, 0.6, case["M"]))


def _batch_shapes(case):
    """(M, kmax) of a batch's instances: part of the case, the same for every seed."""
    rng = np.random.default_rng([case["n"], case["M_lo"], case["M_hi"]])
    return [(int(rng.integers(case["M_lo"], case["M_hi"] + 1)), int(rng.integers(2, 6))) for _ in range(case["n"])]


def _batch_inputs(case, seed):
    rng = np.random.default_rng([seed, case["n"], 2])
    return [(_covariance(*_state(M, rng, (0.5, 1.5), (0.2, 0.6))), k) for M, k in _batch_shapes(case)]


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _spin_table(case, seed):
    """The sampler's input in plain torch, so that it does not depend on the package's kernels."""
    return _table(_cuda(_V(case, seed)[0]), case["K"], "spin_cumulants")


def _uniforms(case, seed):
    g = torch.Generator().manual_seed(seed * 7 + case["M"])
    return torch.rand(case["n"], case["M"], dtype=torch.float64, generator=g).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fit":
        U, r, eta, V_target = _fit_inputs(case, seed)
        M, K = case["M"], case["kmax"]
        return {"kind": kind, "U": _cuda(U), "r": _cuda(r).requires_grad_(), "eta": _cuda(eta).requires_grad_(),
                "kmax": K, "target": gbs.cumulants(_cuda(V_target), K), "w": gbs.fit_weights(M, K, "cuda")}
    if kind == "batch":
        inst = _batch_inputs(case, seed)
        return {"kind": kind, "batch": gbs.Batch([_cuda(V) for V, _ in inst], [k for _, k in inst], case["precision"])}
    if kind == "sample":
        M, K, batch, prec = case["M"], case["K"], case["batch"], case["precision"]
        return {"kind": kind, "kappa": _spin_table(case, seed), "u": _uniforms(case, seed),
                "ws": torch.empty(gbs.sampler_workspace_bytes(M, K, batch, prec), dtype=torch.uint8, device="cuda"),
                **{k: case[k] for k in ("M", "K", "batch", "precision")}}
    V, mean = _V(case, seed)
    s = dict(case, V=_cuda(V), mean=_cuda(mean))
    if kind != "call":
        prec = case.get("precision", "fp64")
        s["out"] = torch.empty(gbs.table_size(case["M"], case["kmax"]), dtype=torch.float64, device="cuda")
        s["ws"] = gbs.Workspace(case["M"], case["kmax"], prec)
    return s


def run(s):
    kind = s["kind"]
    if kind == "call":
        return getattr(gbs, s["fn"])(s["V"], s["kmax"], s["precision"])
    if kind == "table":
        return getattr(gbs, s["fn"])(s["V"], s["kmax"], s["precision"], out=s["out"], workspace=s["ws"], check=False)
    if kind == "displaced":
        return gbs.displaced_tables(s["V"], s["mean"], s["kmax"], s["table"], out=s["out"], workspace=s["ws"], check=False)
    if kind == "fit":
        s["r"].grad = s["eta"].grad = None
        kt = gbs.CumulantFn.apply(gbs.CovarianceFn.apply(s["r"], s["eta"], s["U"]), s["kmax"])
        loss = (s["w"] * (kt - s["target"]) ** 2).sum()
        loss.backward()
        return {"loss": loss.detach(), "grad_r": s["r"].grad, "grad_eta": s["eta"].grad, "kappa": kt.detach()}
    if kind == "batch":
        return s["batch"].run()
    bits, logp, q0 = gbs.sample(s["kappa"], s["M"], s["K"], u=s["u"], batch=s["batch"], precision=s["precision"],
                                want_q0=True, workspace=s["ws"], check=False)
    return {"bits": bits, "logp": logp, "q0": q0}


def _table_work(M, kmax):
    """A table needs its determinants' leaf step (22 multiply-adds) and 2^{d-1} products per entry."""
    n = sum(comb(M, d) for d in range(1, kmax + 1))
    return 8.0 * (n + 4 * M * M), sum(2.0 * comb(M, d) * (22 + 2 ** (d - 1)) for d in range(1, kmax + 1))


def work(case):
    kind, M = case["kind"], case.get("M", 0)
    if kind == "batch":
        each = [_table_work(m, k) for m, k in _batch_shapes(case)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    if kind == "sample":
        K, n, es = case["K"], case["n"], 4 if case["precision"] == "fp32" else 8
        nk = sum(comb(M, d) for d in range(1, K + 1))
        # every cumulant of order K once per sample, and the p1 / p2 tables once over each later bit
        tables = comb(M, 4) if K == 5 else comb(M, 3)
        return {"bytes": 8.0 * nk + n * (9.0 * M + 8 * M), "flops": 2.0 * n * (comb(M, K) + 3.0 * tables)}
    b, f = _table_work(M, case["kmax"])
    if kind == "fit":  # the table, its target, the weights, and the adjoint's P0 and gradient over the same entries
        return {"bytes": 3 * b + 16.0 * M * M, "flops": 3 * f}
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same values in plain torch, 64 bits

def _binoms(M, device):
    n = torch.arange(M + 1, dtype=torch.int64)
    cols = [torch.ones_like(n)]
    for k in range(1, 6):
        cols.append(torch.tensor([comb(int(x), k) for x in n], dtype=torch.int64))
    return [c.to(device) for c in cols]


def _subsets(M, d, device):
    """All d-subsets in colex order, one column of ascending modes each: (d, C(M, d))."""
    if d == 0:
        return torch.zeros((0, 1), dtype=torch.int16, device=device)
    low = _subsets(M, d - 1, device)
    return torch.cat([torch.cat([low[:, : comb(c, d - 1)], torch.full((1, comb(c, d - 1)), c, dtype=torch.int16, device=device)])
                      for c in range(d - 1, M)], dim=1)


def _p0_of(A, half_mean, cols, M):
    """det(A_T)^{-1/2}, with exp(-b_T A_T^{-1} b_T) for first moments, of the subsets in cols (list of index vectors)."""
    rows = [c for x in cols for c in (x, x + M)]
    n = len(rows)
    L = [[None] * n for _ in range(n)]
    prod, quad, y = None, None, []
    for k in range(n):
        dkk = A[rows[k], rows[k]]
        for m in range(k):
            dkk = dkk - L[k][m] * L[k][m]
        inv = dkk.rsqrt()
        prod = inv if prod is None else prod * inv
        for r in range(k + 1, n):
            v = A[rows[r], rows[k]]
            for m in range(k):
                v = v - L[r][m] * L[k][m]
            L[r][k] = v * inv
        if half_mean is not None:
            b = half_mean[rows[k]]
            for m in range(k):
                b = b - L[k][m] * y[m]
            y.append(b * inv)
            quad = y[-1] ** 2 if quad is None else quad + y[-1] ** 2
    return prod if half_mean is None else prod * torch.exp(-quad)


def _table(V, kmax, fn, mean=None):
    """One table from the definitions: determinants, then sums over the subsets of each S."""
    M, dev = V.shape[0] // 2, V.device
    A = 0.5 * (V + torch.eye(2 * M, dtype=V.dtype, device=dev))
    hm = None if mean is None else 0.5 * mean
    B = _binoms(M, dev)
    low_sets = [_subsets(M, d, dev) for d in range(kmax)]
    p0, ky, out = [None], [None], []
    for d in range(1, kmax + 1):
        P, Y, W = [], [], []
        c0 = d - 1
        while c0 < M:  # chunks of whole top modes
            c1, n = c0, 0
            while c1 < M and (n == 0 or n + comb(c1, d - 1) <= 16_000_000):
                n += comb(c1, d - 1)
                c1 += 1
            top = torch.cat([torch.full((comb(c, d - 1),), c, dtype=torch.int64, device=dev) for c in range(c0, c1)])
            low = torch.cat([low_sets[d - 1][:, : comb(c, d - 1)] for c in range(c0, c1)], dim=1)
            cols = [x.long() for x in low] + [top]
            c0 = c1
            p = _p0_of(A, hm, cols, M)

            def at(tabs, mask):  # a lower-order table at the subset of S that mask selects
                if not mask:
                    return 1.0
                pos = [i for i in range(d) if mask >> i & 1]
                if len(pos) == d:
                    return p
                return tabs[len(pos)][sum(B[i + 1][cols[e]] for i, e in enumerate(pos))]

            full = (1 << d) - 1
            if fn == "vacuum_probs":
                w = p
            elif fn == "click_moments":
                w = sum((-1) ** bin(t).count("1") * at(p0, t) for t in range(1, full + 1)) + 1.0
            elif fn == "spin_correlators":
                w = (-1) ** d * (1.0 + sum((-2.0) ** bin(t).count("1") * at(p0, t) for t in range(1, full + 1)))
            else:  # cumulants of the no-click indicators, by the block that holds the lowest mode
                y = p
                for R in range(1, full, 2):
                    y = y - at(ky, R) * at(p0, full ^ R)
                Y.append(y)
                if fn == "cumulants":
                    w = 1.0 - p if d == 1 else (-1.0) ** d * y
                else:
                    w = 2.0 * p - 1.0 if d == 1 else 2.0 ** d * y
            if d < kmax:
                P.append(p)
            W.append(w)
        if d < kmax:
            p0.append(torch.cat(P))
            ky.append(torch.cat(Y) if Y else None)
        out += W
    return torch.cat(out)


def _sample(kappa, M, K, u):
    """The chain-rule sampler, every table entry over n bits multiplied by 2^n. Tables in [..][sample] layout;
    Q[a][l] = p+(x_{a-1}..x_l) (1 for l = a, 0 above), R1[a][e] = p1(x_a..~x_e..x_1), T[a] = p2 symmetric in the
    two elided bits; bit a elided from its own row is the row below."""
    S, dev = u.shape[0], u.device
    f8 = dict(dtype=torch.float64, device=dev)
    off = [0, 0]
    for d in range(1, K + 1):
        off.append(off[-1] + comb(M, d))

    def seg(d, base, n):
        return kappa[off[d] + base: off[d] + base + n]

    chi = torch.ones(M + 2, S, **f8)
    P = torch.ones(M + 1, S, **f8)
    Q = torch.zeros(M + 2, M + 2, S, **f8)
    R1 = torch.zeros(M + 1, M + 1, S, **f8)
    T = torch.zeros(M + 1, M + 1, M + 1, S, **f8) if K > 3 else None
    Z4, Z5 = {}, {}
    bits = torch.zeros(S, M, dtype=torch.uint8, device=dev)
    q0 = torch.zeros(S, M, **f8)
    Q[1, 1] = 1.0
    opp, op1, op2 = {3: (2, 2, 1), 4: (2, 2, 1), 5: (3, 3, 2)}[K]
    for n in range(1, M + 1):
        m = n - 1
        k1 = kappa[n - 1]
        k2 = seg(2, comb(m, 2), m)[:, None]                    # kappa(i, n), i = 1..m
        tri = torch.tril_indices(m, m, -1, device=dev)         # pairs j < i in colex order
        k3 = torch.zeros(m, m, **f8)
        k3[tri[0], tri[1]] = seg(3, comb(m, 3), comb(m, 2))
        x = chi[1:n]
        up = Q[n, 2:n + 1]                                     # p+(x_{n-1}..x_{i+1}), i = 1..m
        B = k1 * P[m]
        if m:
            B = B + (k2 * x * R1[m, 1:n]).sum(0)
        if K == 3:
            if m >= 2:
                B = B + (x * up * torch.einsum("ij,ijs->is", k3, R1[0:m, 1:n] * x[None])).sum(0)
        elif m >= 2:
            e, d = tri[0] + 1, tri[1] + 1
            W = T[m][e, d] * chi[e] * chi[d]
            D = comb(m, 2)
            B = B + seg(3, comb(m, 3), D) @ W
            later = torch.arange(n + 1, M + 1)                 # this W's part of every later bias
            if len(later):
                base = torch.tensor([off[4] + comb(int(q) - 1, 4) + comb(m, 3) for q in later], device=dev)
                Z4[n] = kappa[base[:, None] + torch.arange(D, device=dev)] @ W
                if K == 5 and len(later) > 1:
                    base = torch.tensor([off[5] + comb(q - 1, 5) + comb(i - 1, 4) + comb(m, 3)
                                         for q in range(n + 2, M + 1) for i in range(n + 1, q)], device=dev)
                    Z5[n] = kappa[base[:, None] + torch.arange(D, device=dev)] @ W
            for i in range(3, n):
                z = Z4[i][n - i - 1]
                if K == 5 and i > 3:
                    z = z + torch.stack([chi[j] * Q[i, j + 1] * Z5[j][comb(n - j - 1, 2) + i - j - 1]
                                         for j in range(3, i)]).sum(0)
                B = B + x[i - 1] * up[i - 1] * z
        a, b = P[m] + B, P[m] - B
        ca, cb = a.clamp_min(0), b.clamp_min(0)
        q = torch.where(ca + cb > 0, ca / (ca + cb), torch.full_like(ca, 0.5))
        one = u[:, m] >= q
        bits[:, m], q0[:, m] = one.to(torch.uint8), q
        chi[n] = torch.where(one, -1.0, 1.0)
        P[n] = torch.where(one, b, a)
        c = chi[n]
        h = 1.0 + k1 * c
        Q[n + 1, n + 1] = 1.0
        if not m:
            Q[2, 1] = h
            R1[1, 1] = P[0]
            continue
        g = k2 * x * c
        new = h * Q[n, 1:n + 1]                                # p+(x_n..x_l), l = 1..n
        new[:m] += torch.einsum("is,ils->ls", g * up, Q[1:n, 1:n])
        new[m] = h
        if opp >= 3:
            v = c * x * torch.einsum("ij,is,ijs->js", k3, x * up, Q[1:n, 2:n + 1])
            new[:m] += torch.einsum("js,jls->ls", v, Q[1:n, 1:n])
        Q[n + 1, 1:n + 1] = new
        r1 = h * R1[m, 1:n]
        if K == 3:
            U = torch.tril(torch.ones(m, m, **f8), -1)[:, :, None] * R1[0:m, 1:n]
            r1 = r1 + up * torch.einsum("eis,is->es", U, g) + torch.einsum("ies,is->es", U, g * up)
        else:
            r1 = r1 + torch.einsum("eis,is->es", T[m][1:n, 1:n], g)
            if op1 >= 3:
                sym = k3 + k3.T
                for i in range(2, n):
                    t = T[i - 1][1:i, 1:i]
                    kx = k3[i - 1, : i - 1, None] * x[: i - 1]
                    r1[: i - 1] += c * x[i - 1] * up[i - 1] * torch.einsum("ejs,js->es", t, kx)
                    pairs = sym[: i - 1, : i - 1].triu(1)[:, :, None] * x[: i - 1, None] * x[None, : i - 1]
                    r1[i - 1] += c * up[i - 1] * (pairs * t).sum((0, 1))
            new = h * T[m][1:n, 1:n]
            if op2 >= 2:
                low = torch.zeros_like(new)                    # [e][d], d < e
                for i in range(2, n):
                    t = T[i - 1][1:i, 1:i]
                    low[: i - 1, : i - 1] += g[i - 1] * up[i - 1] * t
                    low[i - 1, : i - 1] += up[i - 1] * torch.einsum("dis,is->ds", t, g[: i - 1])
                low = torch.tril(torch.ones(m, m, **f8), -1)[:, :, None] * low
                new = new + low + low.transpose(0, 1)
            T[n][1:n, 1:n] = new
            T[n][n, 1:n] = T[n][1:n, n] = R1[m, 1:n]
        R1[n, 1:n] = r1
        R1[n, n] = P[m]
    logp = torch.log(P[M]) - M * math.log(2.0)
    return {"bits": bits, "logp": logp, "q0": q0}


def exact(case, seed):
    kind = case["kind"]
    if kind == "sample":
        M, K, n = case["M"], case["K"], case["n"]
        # steps of a python loop, and the sampler's own operations in 64 bits: past these it takes too long
        if (K > 3 and (M > 100 or M ** 4 * n > 3e10)) or (K == 3 and M ** 3 * n > 5e11):
            return None
        got = _sample(_spin_table(case, seed), M, K, _uniforms(case, seed))
        got["bits"] = None  # a draw, not a rounded number
        return got
    if kind == "batch":
        return [_table(_cuda(V), k, "cumulants") for V, k in _batch_inputs(case, seed)]
    if kind == "fit":
        U, r, eta, V_target = _fit_inputs(case, seed)
        target = _table(_cuda(V_target), case["kmax"], "cumulants")
        U, r, eta = _cuda(U), _cuda(r).requires_grad_(), _cuda(eta).requires_grad_()
        S = torch.cat([torch.cat([U.real, -U.imag], 1), torch.cat([U.imag, U.real], 1)], 0)
        e2, q = torch.cat([eta, eta]), torch.exp(torch.cat([-2 * r, 2 * r]))
        V = e2.sqrt()[:, None] * ((S * q) @ S.T) * e2.sqrt() + torch.diag(1 - e2)
        kt = _table(V, case["kmax"], "cumulants")
        w = torch.cat([torch.full((comb(case["M"], d),), 1.0 / comb(case["M"], d), dtype=torch.float64, device="cuda")
                       for d in range(1, case["kmax"] + 1)])
        loss = (w * (kt - target) ** 2).sum()
        loss.backward()
        return {"loss": loss.detach(), "grad_r": r.grad, "grad_eta": eta.grad, "kappa": kt.detach()}
    V, mean = _V(case, seed)
    if kind == "displaced":
        fn = {"p0": "vacuum_probs", "mu": "click_moments", "kappa": "cumulants", "spin_c": "spin_correlators",
              "spin_kappa": "spin_cumulants"}[case["table"]]
        return _table(_cuda(V), case["kmax"], fn, _cuda(mean))
    return _table(_cuda(V), case["kmax"], case["fn"])
