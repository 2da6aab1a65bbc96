"""Performance cases: the work users of this framework have it do.

A case is one of three calls a DMRG program makes:

- "sigma": sigma = H_eff psi at a middle bond (dmrg_sigma), the inner product
  of every solver, in each arithmetic (FP64, BF16X2, BF16X3, FP16X2) and with
  device or host buffers;
- "davidson": a lowest-eigenpair solve of a fixed number of products
  (dmrg_davidson), what the serving loop and the sweeps run. With synthetic
  operators only FP64 at small sizes: their diagonal is dense around the
  first Ritz values, so the preconditioner amplifies any rounding (a 1e-7
  product gives another vector after 4 products at K=36, M=500). Mixed
  solves are measured inside the sweeps, where they converge;
- "sweep": initial blocks from integrals and two-site sweeps
  (dmrg_build_blocks + dmrg_sweep), NC or mixed NC/CN.

Sizes are those of the repository's configurations: K in {8 .. 108} spatial
orbitals, bond dimensions 60 .. 4000, N between K/2 and K electrons (30 for
the K=108 middle bond), 2Sz = N mod 2. Middle-bond operators are the
library's synthetic ones (dmrg_load_synthetic: seeded N(0,1) blocks over the
sector structure). Contexts use the defaults a solver meets: no autotuning.

exact() restates the same numbers in plain torch, in 64 bits, from the
published definitions of the operator layout and of the counter-based
generator, without the library.
"""

import math

import numpy as np
import torch

PRECS = ("fp64", "bf16x2", "bf16x3", "fp16x2")
CODE = {"fp64": 0, "bf16x2": 1, "bf16x3": 2, "fp16x2": 3}   # dmrg_prec
SPLIT_BYTES = {"fp64": 8, "bf16x2": 4, "bf16x3": 6, "fp16x2": 4}  # per operator element


def listed():
    def sigma(name, prec, K, N, M, buffers="device"):
        return {"name": name, "call": "sigma", "prec": prec, "K": K, "N": N, "M": M, "buffers": buffers}

    def solve(name, prec, K, N, M, products):
        return {"name": name, "call": "davidson", "prec": prec, "K": K, "N": N, "M": M, "products": products}

    def sweep(name, prec, K, N, M, cut):
        return {"name": name, "call": "sweep", "prec": prec, "K": K, "N": N, "M": M, "cut": cut, "sweeps": 2}

    return [
        # the first steps of any sweep and unit-test sized problems: launches and latency
        sigma("sigma_fp64_k8_m64", "fp64", 8, 8, 64),
        # one product of a mid-sized serving request in the reference arithmetic, odd N and M
        sigma("sigma_fp64_k36_m501", "fp64", 36, 27, 501),
        # a larger serving request, FP64: also the energy of every mixed-precision solve of this size
        sigma("sigma_fp64_k54_m1000", "fp64", 54, 37, 1000),
        # the repository's benchmark workload (K=108 middle bond, M=2000), FP64
        sigma("sigma_fp64_k108_m2000", "fp64", 108, 30, 2000),
        # small serving request through host buffers, as a program that keeps psi on the host calls it
        sigma("sigma_fp16x2_k24_m250_host", "fp16x2", 24, 17, 250, "host"),
        # mid-sized serving request in the fastest bf16 mode
        sigma("sigma_bf16x2_k54_m1000", "bf16x2", 54, 41, 1000),
        # FeMoco-shaped orbital count in the 24-bit mode
        sigma("sigma_bf16x3_k76_m2000", "bf16x3", 76, 57, 2000),
        # the benchmark workload in the production arithmetic
        sigma("sigma_fp16x2_k108_m2000", "fp16x2", 108, 30, 2000),
        # the largest bond dimension served
        sigma("sigma_fp16x2_k76_m4000", "fp16x2", 76, 60, 4000),
        # a reference-arithmetic solve of a small request
        solve("davidson_fp64_k24_m250", "fp64", 24, 19, 250, 16),
        # a small molecule at full precision: all steps of the method, NC partition
        sweep("sweep_fp64_k8_m100_nc", "fp64", 8, 8, 100, -1),
        # production sweeps: solves with the mixed sigma, mixed NC/CN partition with the cut in the middle
        sweep("sweep_fp16x2_k16_m150_mixed", "fp16x2", 16, 15, 150, 8),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choices(("sigma", "davidson", "sweep"), (0.7, 0.2, 0.1))[0]
    if call == "sweep":
        K = rng.randrange(6, 13, 2)
        return {"call": "sweep", "prec": rng.choice(PRECS), "K": K, "N": rng.randint(K // 2, K),
                "M": log_int(30, 150), "cut": rng.choice((-1, K // 2)), "sweeps": 2}
    while True:
        if call == "davidson":
            K = 2 * log_int(4, 12)
            return {"call": call, "prec": "fp64", "K": K, "N": rng.randint(K // 2, K), "M": log_int(60, 250),
                    "products": rng.randint(4, 16)}
        prec = rng.choice(PRECS)
        K = 2 * log_int(4, 54)
        case = {"call": call, "prec": prec, "K": K, "N": 30 if K > 90 else rng.randint(K // 2, K),
                "M": log_int(60, 4000), "buffers": rng.choice(("device", "device", "host"))}
        flops, elements = _cost(case)
        if elements <= 4.2e9 and flops <= (5.6e11 if prec == "fp64" else 2.2e12):  # at most the largest listed ones
            return case


# ---------------------------------------------------------------- problems
def sectors(K, N, M):
    """(N, 2Sz, dim) lists of the two sides: dimensions follow a Gaussian of
    widths 3 and 2 about (N/2, 2Sz/2), rounded to sum to M."""
    ns, sz = K // 2, N % 2
    cand = []
    for n in range(N + 1):
        nr = N - n
        if n > 2 * ns or nr > 2 * ns:
            continue
        top, topr = min(n, 2 * ns - n), min(nr, 2 * ns - nr)
        cand += [(n, s) for s in range(-top, top + 1) if (s - n) % 2 == 0 and abs(sz - s) <= topr and (sz - s - nr) % 2 == 0]
    w = np.array([math.exp(-((n - N / 2) ** 2) / 18 - ((s - sz / 2) ** 2) / 8) for n, s in cand])
    exact = M * w / w.sum()
    dims = np.floor(exact).astype(np.int64)
    order = sorted(range(len(cand)), key=lambda a: (-(exact[a] - dims[a]), cand[a]))
    for a in order[:int(M - dims.sum())]:
        dims[a] += 1
    left = sorted((n, s, int(d)) for (n, s), d in zip(cand, dims) if d > 0)
    return left, sorted((N - n, sz - s, d) for n, s, d in left)


def _spin(p):
    return 1 if p % 2 == 0 else -1


def _operators(nL, n):
    """Canonical operators of both sides: key -> (shift, symmetric)."""
    left = {"H": ((0, 0), True)}
    left.update({("cd", p): ((1, _spin(p)), False) for p in range(nL)})
    left.update({("RL", p): ((-1, -_spin(p)), False) for p in range(nL, n)})
    right = {"H": ((0, 0), True)}
    right.update({("d", p): ((-1, -_spin(p)), False) for p in range(nL, n)})
    right.update({("RR", p): ((-1, -_spin(p)), False) for p in range(nL)})
    for p in range(nL):
        for r in range(p + 1, nL):
            s = _spin(p) + _spin(r)
            left["A", p, r], right["P", p, r] = ((2, s), False), ((-2, -s), False)
    for p in range(nL):
        for q in range(p, nL):
            s = _spin(p) - _spin(q)
            left["B", p, q], right["Q", p, q] = ((0, s), p == q), ((0, -s), p == q)
    return left, right


def _terms(nL, n):
    """(left key, left transposed, right key, right transposed, coefficient, right parity)."""
    out = [("H", False, None, False, 1.0, 0), (None, False, "H", False, 1.0, 0)]
    for p in range(nL):
        out += [(("cd", p), False, ("RR", p), False, 1.0, 1), (("cd", p), True, ("RR", p), True, -1.0, 1)]
    for p in range(nL, n):
        out += [(("RL", p), True, ("d", p), False, 1.0, 1), (("RL", p), False, ("d", p), True, -1.0, 1)]
    for p in range(nL):
        for r in range(p + 1, nL):
            out += [(("A", p, r), False, ("P", p, r), False, 1.0, 0), (("A", p, r), True, ("P", p, r), True, 1.0, 0)]
    for p in range(nL):
        for q in range(nL):
            k = (p, q) if p <= q else (q, p)
            out.append((("B",) + k, p > q, ("Q",) + k, p > q, 1.0, 0))
    return out


class _Side:
    """Sector dimensions and the flat store offset of every operator block."""

    def __init__(self, secs, ops, base):
        self.dim = {(n, s): d for n, s, d in secs}
        self.ops, self.start = ops, {}
        self.rel = {}   # shift -> {input sector: offset within the operator}
        for dq, _ in set(ops.values()):
            at, off = {}, 0
            for q in sorted(self.dim):
                qo = (q[0] + dq[0], q[1] + dq[1])
                if qo in self.dim:
                    at[q] = off
                    off += self.dim[q] * self.dim[qo]
            self.rel[dq] = (at, off)
        for k, (dq, _) in ops.items():
            self.start[k] = base
            base += self.rel[dq][1]
        self.end = base


class _Model:
    """Terms grouped by (shifts, transpositions, symmetry, coefficient): one batched contraction per group and psi block."""

    def __init__(self, case):
        K, self.N, self.sz = case["K"], case["N"], case["N"] % 2
        left, right = sectors(K, self.N, case["M"])
        ol, orr = _operators(K, 2 * K)
        self.L = _Side(left, ol, 0)
        self.R = _Side(right, orr, self.L.end)
        self.elements = self.R.end
        self.groups = {}
        for kl, tl, kr, tr, c, par in _terms(K, 2 * K):
            key = (ol[kl] if kl else None, tl, orr[kr] if kr else None, tr, c, par)
            self.groups.setdefault(key, []).append((kl, kr))
        self.blocks, off = [], 0
        for q in sorted(self.L.dim):
            qr = (self.N - q[0], self.sz - q[1])
            if qr in self.R.dim:
                self.blocks.append((q, qr, self.L.dim[q], self.R.dim[qr], off))
                off += self.L.dim[q] * self.R.dim[qr]
        self.size = off
        self.at = {b[0]: b for b in self.blocks}

    def products(self):
        """(group key, pairs, input block, output block)."""
        for key, pairs in self.groups.items():
            (dl, tl), (dr, tr) = ((k[0] if k else (0, 0), t) for k, t in ((key[0], key[1]), (key[2], key[3])))
            for b in self.blocks:
                q = tuple(x - y if tl else x + y for x, y in zip(b[0], dl))
                qr = tuple(x - y if tr else x + y for x, y in zip(b[1], dr))
                o = self.at.get(q)
                if o is not None and o[1] == qr:
                    yield key, pairs, b, o

    def flops(self):
        total = 0.0
        for key, pairs, (_, _, m, n, _), (_, _, mo, no, _) in self.products():
            one = (2 * m * n * no if key[0] is None else 2 * mo * m * n if key[2] is None else
                   min(2 * mo * m * n + 2 * mo * n * no, 2 * m * n * no + 2 * mo * m * no))
            total += len(pairs) * float(one)
        return total


_COST = {}


def _cost(case):
    """(flops of one product, stored operator elements)."""
    k = (case["K"], case["N"], case["M"])
    if k not in _COST:
        m = _Model(case)
        _COST[k] = (m.flops(), m.elements, m.size)
    return _COST[k][:2]


def _psi(size, seed):
    x = np.random.default_rng(seed).standard_normal(size)
    return x / np.linalg.norm(x)


def _integrals(K, seed):
    """t symmetric N(0, 1) and v with the 8-fold symmetry N(0, 0.1^2), both decaying with orbital distance."""
    rng = np.random.default_rng(seed)
    d = np.exp(-np.abs(np.subtract.outer(np.arange(K), np.arange(K))) / 8.0)
    t = rng.standard_normal((K, K))
    t = (t + t.T) / 2 ** 0.5 * d
    v = 0.1 * rng.standard_normal((K, K, K, K))
    v = (v + v.transpose(1, 0, 2, 3)) / 2 ** 0.5
    v = (v + v.transpose(0, 1, 3, 2)) / 2 ** 0.5
    v = (v + v.transpose(2, 3, 0, 1)) / 2 ** 0.5
    return t, np.ascontiguousarray(v * d[:, :, None, None] * d[None, None, :, :])


# ------------------------------------------------------------------ running
class _Ctx:
    """A library context that goes with its state."""

    def __init__(self, **opts):
        from paper_2103_09976_gb300 import capi
        self.capi, self.h = capi, capi.dmrg_create(device=0, **opts)

    def __del__(self):
        if getattr(self, "h", None) is not None:
            self.capi.dmrg_destroy(self.h)
            self.h = None


def prepare(case, seed):
    from paper_2103_09976_gb300 import capi
    if case["call"] == "sweep":
        return {"case": case, "seed": seed, "tv": _integrals(case["K"], seed)}
    opts = {"sigma_prec": CODE[case["prec"]]}
    if case["call"] == "davidson":
        opts["dav_max_iter"] = case["products"]
    ctx = _Ctx(**opts)
    left, right = sectors(case["K"], case["N"], case["M"])
    capi.dmrg_load_synthetic(ctx.h, case["K"], 2 * case["K"], case["N"], case["N"] % 2, left, right, seed)
    x = _psi(capi.dmrg_psi_layout(ctx.h)["size"], seed)
    y = np.zeros_like(x)
    if case.get("buffers") != "host":
        x, y = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    return {"case": case, "ctx": ctx, "x": x, "y": y}


def run(state):
    from paper_2103_09976_gb300 import capi
    case = state["case"]
    if case["call"] == "sigma":
        capi.dmrg_sigma(state["ctx"].h, -1, state["x"], state["y"])
        return state["y"]
    if case["call"] == "davidson":
        # the tolerance is never reached: a fixed number of products
        e, products, _ = capi.dmrg_davidson(state["ctx"].h, -1, state["x"], 1e-30, state["y"])
        # the sign of an eigenvector is arbitrary: the one on the guess's side
        sign = torch.sign(torch.dot(state["x"], state["y"]))
        return {"energy": np.array([e]), "psi": state["y"] * sign, "products": products}
    K, M = case["K"], case["M"]
    t, v = state["tv"]
    ctx = _Ctx(sigma_prec=CODE[case["prec"]], mixed_cut=case["cut"], seed=state["seed"])
    capi.dmrg_build_blocks(ctx.h, t, v, K, case["N"], case["N"] % 2, M)
    energies, discarded = capi.dmrg_sweep(ctx.h, [M] * case["sweeps"], 1e-9 if case["prec"] == "fp64" else 1e-7)
    log = capi.dmrg_sweep_log(ctx.h)
    out = {"energies": energies, "discarded": discarded, "steps": np.array([s["energy"] for s in log])}
    if case["prec"] == "fp64":
        # an operator the sweep leaves behind: H of the right block of two orbitals. Its basis are singular vectors
        # of psi, which near-equal singular values rotate by more than a mixed solve's error
        out["block"] = capi.dmrg_block_read(ctx.h, 1, K - 2, 0)
    return out


def work(case):
    flops, elements = _cost(case)
    size = _COST[case["K"], case["N"], case["M"]][2]
    if case["call"] == "sigma":
        return {"bytes": SPLIT_BYTES[case["prec"]] * elements + 16 * size, "flops": flops}
    if case["call"] == "davidson":  # the operators exceed the caches: each product reads them
        return {"bytes": case["products"] * (SPLIT_BYTES[case["prec"]] * elements + 16.0 * size),
                "flops": case["products"] * flops}
    # two products per step and the operators of its bond written and read once, taking the middle bond for half the steps
    steps = case["sweeps"] * (case["K"] - 1) / 2
    return {"bytes": steps * 16.0 * elements, "flops": steps * 2 * flops}


def tolerance(case):
    if case["call"] == "sigma":
        # about four times the distance of each arithmetic from exact() at the largest listed sizes. FP64: sums of up to
        # 1e6 products; mixed: operands of 16 (BF16X2), 24 (BF16X3) and 22 (FP16X2) bits, products and sums in FP32
        return {"fp64": {"rel": 4e-14, "max": 4e-13}, "bf16x2": {"rel": 2.5e-5, "max": 2.5e-4},
                "bf16x3": {"rel": 4e-6, "max": 4e-5}, "fp16x2": {"rel": 4e-6, "max": 4e-5}}[case["prec"]]
    if case["call"] == "davidson":
        # rounding of a product (1e-15) grows with the products: psi was 1e-10 to 4e-7 off exact()
        return {"rel": 4e-5, "max": 4e-4}
    # steps converge to |r|^2 < 1e-9 (FP64) or 1e-7; energies of two mixed arithmetics differ by 2e-6, discarded weights by 5e-5
    return {"rel": 1e-5, "max": 1e-4} if case["prec"] == "fp64" else {"rel": 2e-4, "max": 2e-3}


# -------------------------------------------------------------------- exact
def _mix(z):
    def shr(a, k):
        return (a >> k) & ((1 << (64 - k)) - 1)

    def signed(c):
        return c - (1 << 64) if c >= 1 << 63 else c
    z = (z ^ shr(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * signed(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _normal(seed, g):
    """Box-Muller numbers of the SplitMix64 counters 2g and 2g + 1 (the published generator)."""
    gamma = 0x9E3779B97F4A7C15 - (1 << 64)

    def u(c):
        return (((_mix((c + 1) * gamma + seed) >> 11) & ((1 << 53) - 1)).double() + 1.0) * 2.0 ** -53
    return torch.sqrt(-2.0 * torch.log(u(2 * g))) * torch.cos(2.0 * math.pi * u(2 * g + 1))


class _Exact:
    def __init__(self, case, seed):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.m, self.seed = _Model(case), seed

    def _blocks(self, side, keys, kind, trans, qin, qout):
        """Used matrices [len(keys), dim(qout), dim(qin)] of the operators `keys`, all of one kind."""
        dq, sym = kind
        qi = qout if trans else qin                      # the stored block's input sector
        qo = (qi[0] + dq[0], qi[1] + dq[1])
        r, c = side.dim[qo], side.dim[qi]
        base = torch.tensor([side.start[k] for k in keys], device=self.dev) + side.rel[dq][0][qi]
        i, j = torch.arange(r, device=self.dev)[:, None], torch.arange(c, device=self.dev)[None, :]
        e = torch.minimum(i, j) * c + torch.maximum(i, j) if sym else i * c + j
        x = _normal(self.seed, base[:, None, None] + e[None])
        return x.transpose(1, 2) if trans else x

    def chunks(self):
        for key, pairs, b, o in self.m.products():
            step = max(1, int(4e7 / max(1, b[2] * o[2] + b[3] * o[3])))
            sign = -key[4] if key[5] and b[0][0] % 2 else key[4]
            for k in range(0, len(pairs), step):
                part = pairs[k:k + step]
                L = self._blocks(self.m.L, [p[0] for p in part], key[0], key[1], b[0], o[0]) if key[0] else None
                R = self._blocks(self.m.R, [p[1] for p in part], key[2], key[3], b[1], o[1]) if key[2] else None
                yield b, o, sign, L, R

    def sigma(self, x):
        y = torch.zeros_like(x)
        for b, o, sign, L, R in self.chunks():
            X = x[b[4]:b[4] + b[2] * b[3]].view(b[2], b[3])
            T = len(L) if L is not None else len(R)
            if L is not None:
                X = (L.reshape(T * o[2], b[2]) @ X).view(T, o[2], b[3]).permute(1, 0, 2).reshape(o[2], T * b[3])
            if R is not None:
                X = X @ R.permute(1, 0, 2).reshape(o[3], T * b[3]).T if L is not None else X @ R.sum(0).T
            elif T > 1:
                X = X.view(o[2], T, b[3]).sum(1)
            y[o[4]:o[4] + o[2] * o[3]] += sign * X.reshape(-1)
        return y

    def diagonal(self):
        d = torch.zeros(self.m.size, dtype=torch.float64, device=self.dev)
        for b, o, sign, L, R in self.chunks():
            if b[0] != o[0]:
                continue
            one = torch.ones(1, dtype=torch.float64, device=self.dev)
            l = torch.diagonal(L, dim1=1, dim2=2) if L is not None else one.expand(len(R), b[2])
            r = torch.diagonal(R, dim1=1, dim2=2) if R is not None else one.expand(len(L), b[3])
            d[b[4]:b[4] + b[2] * b[3]] += sign * (l.T @ r).reshape(-1)
        return d

    def davidson(self, x, products):
        """The documented steps: diagonal preconditioner clamped at 1e-8, Gram-Schmidt twice; fewer products than the space holds."""
        diag = self.diagonal()
        V, AV = [x / x.norm()], []
        while True:
            AV.append(self.sigma(V[-1]))
            v, a = torch.stack(V), torch.stack(AV)
            h = v @ a.T
            w, Y = torch.linalg.eigh(((h + h.T) / 2).cpu())
            c = Y[:, 0].to(self.dev)
            y, ay = c @ v, c @ a
            if len(AV) >= products:
                return float(w[0]), y
            den = w[0].to(self.dev) - diag
            den = torch.where(den.abs() < 1e-8, torch.where(den < 0, -1e-8, 1e-8), den)
            t = (ay - float(w[0]) * y) / den
            for _ in range(2):
                t = t - (v @ t) @ v
            V.append(t / t.norm())


def exact(case, seed):
    if case["call"] == "sweep":
        return None
    flops, elements = _cost(case)
    products = case.get("products", 1)
    if products * (flops / 8e11 + elements / 1e9) > 15:
        return None
    e = _Exact(case, seed)
    x = torch.from_numpy(_psi(e.m.size, seed)).to(e.dev)
    if case["call"] == "sigma":
        return e.sigma(x)
    energy, psi = e.davidson(x, products)
    return {"energy": np.array([energy]), "psi": psi * torch.sign(torch.dot(psi, x)), "products": None}
