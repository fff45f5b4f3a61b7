"""The workloads this library is timed on, and their results in plain 64-bit torch.

A case is one call, or one short sequence of calls, of the public API
(paper_2605_17222_gb300.binding): linear transformations of every algorithm
over the parameter sets of the repository, a batch, a bootstrapping chain, and
the key-switching steps a custom schedule is built from.

  listed()           the standing cases
  draw(rng)          one more case of the same ranges
  prepare(case, s)   context, keys, diagonals and ciphertexts on the GPU
  run(state)         one pass; returns the output residues
  work(case)         bytes and operations a pass cannot do without
  exact(case, s)     the same outputs from the definitions of the steps, in
                     torch int64 arithmetic without this library's code

All inputs are uniform residues: keys, encrypted polynomials and encoded
diagonals are uniform to the arithmetic, whatever they encrypt or encode.
"""
import math

import torch

from paper_2605_17222_gb300 import binding, synth

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def _lt(name, params, level, algo, split, stride=1, offset0=0):
    n1, n2, n3 = split
    return {"name": name, "kind": "lt", "params": params, "level": level, "algo": algo, "n1": n1, "n2": n2,
            "n3": n3, "stride": stride, "offset0": offset0}


def listed():
    return [
        # the smallest LT a user evaluates (unit tests, functional prototypes): every launch is latency
        _lt("lt-toy", "toy", 4, "th", (4, 4, 4)),
        # un-hoisted BSGS on a mid-size ring: many small key switches one after another
        _lt("lt-n14-bsgs", "n14", 8, "bsgs", (8, 8, 1)),
        # Algorithm 1 with a strided, based window and a partial last digit (an odd level after some rescales)
        _lt("lt-n15-dh", "n15", 11, "dh", (12, 8, 1), stride=3, offset0=-141),
        # the hoisted diagonal method at a prime diagonal count (small dense layers)
        _lt("lt-n15-diag", "n15", 16, "diag", (1, 37, 1)),
        # a deep level of a big ring: short chains, one limb in the last digit
        _lt("lt-n16-low", "n16", 9, "th", (2, 8, 4)),
        # the headline workload: 256 diagonals at N = 2^16, top level, the split the autotuner takes
        _lt("lt-n16-th", "n16", 24, "th", (1, 64, 4)),
        # the paper's Set-A: one dense 4096 x 4096 matrix, 54-bit moduli, the paper's split
        _lt("lt-setA", "setA", 5, "th", (16, 16, 16)),
        # 64-bit-wide moduli on the ring of the paper's Set-B, a convolution-sized window
        _lt("lt-setB", "setB", 16, "th", (4, 8, 8), stride=2, offset0=-250),
        # bootstrapping's CoeffToSlot: three LTs through lt_eval_chain
        {"name": "chain-cts", "kind": "chain", "params": "n16", "level": 24, "radices": "5,5,5", "inverse": True},
        # a serving batch: ciphertexts at mixed levels against one matrix
        {"name": "batch-n16", "kind": "batch", "params": "n16", "level": 24, "level_step": 8, "count": 16,
         "n1": 1, "n2": 64, "n3": 4, "stride": 1, "offset0": 0},
        # one hoisted rotation from the exported steps: Decompose, key inner product, two ModDowns
        {"name": "rotation-n16", "kind": "rotation", "params": "n16", "level": 24, "rot": 5},
        # a forward and an inverse transform of one extended polynomial
        {"name": "ntt-n14", "kind": "ntt", "params": "n14", "level": 8},
    ]


# D up to this many diagonals per parameter set in drawn LTs
_MAX_D = {"toy": 512, "n14": 256, "n14d8": 128, "n15": 256, "n16": 256, "setA": 4096, "setB": 256}
_MAX_KEYS = 80


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def _draw_split(rng, algo, D):
    if algo == "diag":
        return (1, D, 1)
    divs = [d for d in range(1, D + 1) if D % d == 0]
    if algo in ("bsgs", "dh"):
        c = [(a, D // a, 1) for a in divs if a <= 64 and D // a <= 64]
    else:
        c = [(a, b, D // (a * b)) for a in divs if a <= 16 for b in divs if D % (a * b) == 0 and D // (a * b) <= 16]
    c = [s for s in c if sum(s) <= _MAX_KEYS]
    return rng.choice(c) if c else None


def draw(rng):
    while True:
        c = _draw(rng)
        if work(c)["flops"] <= 3e10:  # half of the largest listed case's
            return c


def _draw(rng):
    kind = rng.choices(["lt", "batch", "chain", "rotation", "ntt", "down"], [12, 2, 1, 2, 2, 2])[0]
    if kind == "lt":
        params = rng.choice(sorted(_MAX_D))
        ps = synth.param_set(params)
        algo = rng.choice(["th", "th", "th", "dh", "bsgs", "diag"])
        while True:
            D = _log_int(rng, 1, _MAX_D[params] if algo == "th" else 64)
            split = _draw_split(rng, algo, D)
            if split:
                break
        stride = 1 if rng.random() < 0.5 else rng.randint(1, max(1, (ps.n // 2 - 1) // max(1, D - 1)))
        offset0 = 0 if rng.random() < 0.6 else rng.randint(-(ps.n // 4), ps.n // 4)
        c = _lt("", params, rng.randint(2, ps.L), algo, split, stride, offset0)
        del c["name"]
        return c
    if kind == "batch":
        params = rng.choice(["toy", "n14", "n15", "n16"])
        ps = synth.param_set(params)
        while True:
            D = _log_int(rng, 4, 128)
            split = _draw_split(rng, "th", D)
            if split:
                break
        return {"kind": "batch", "params": params, "level": rng.randint(max(2, ps.L // 2), ps.L),
                "level_step": rng.randint(0, ps.L // 3), "count": rng.randint(2, 12), "n1": split[0],
                "n2": split[1], "n3": split[2], "stride": 1, "offset0": 0}
    if kind == "chain":
        params = rng.choice(["n14", "n15", "n16"])
        ps = synth.param_set(params)
        n = rng.choice([3, 4])
        logs = ps.log_n - 1
        rad = [logs // n + (1 if i < logs % n else 0) for i in range(n)]
        rng.shuffle(rad)
        return {"kind": "chain", "params": params, "level": rng.randint(n + 1, ps.L),
                "radices": ",".join(map(str, rad)), "inverse": rng.random() < 0.5}
    params = rng.choice(["toy", "n14", "n15", "n16", "setA", "setB"])
    ps = synth.param_set(params)
    c = {"kind": kind, "params": params, "level": rng.randint(2, ps.L)}
    if kind == "rotation":
        c["rot"] = rng.randint(1, ps.n // 2 - 1)
    if kind == "down":
        c["op"] = rng.choice(["moddown", "moddown_rescale", "rescale"])
    return c


# ------------------------------------------------------------------ shapes shared by prepare, work and exact
def _stages(case):
    """(offset0, stride, D, split) of each stage of a factored slot DFT, first
    applied first: a group of r radix-2 butterfly levels is one LT whose
    diagonals are the multiples of its first level's half-width."""
    rad = [int(r) for r in case["radices"].split(",")]
    top = synth.param_set(case["params"]).log_n - 1
    out, t = [], 0
    for r in rad:
        h = 1 << t
        t += r
        if t == top:
            out.append((0, h, 1 << r))
        else:
            out.append((-((1 << r) - 1) * h, h, 2 << r))
    return [(o, h, D, (1, D // 2, 2)) for o, h, D in (out[::-1] if case["inverse"] else out)]


def _levels(case):
    """The levels of a batch's ciphertexts (never below 2)."""
    return [max(2, case["level"] - case["level_step"] * (i % 3)) for i in range(case["count"])]


def _lts(case):
    """Every (level, algo, split, stride, offset0, D) that the case evaluates."""
    if case["kind"] == "lt":
        s = (case["n1"], case["n2"], case["n3"])
        return [(case["level"], case["algo"], s, case["stride"], case["offset0"], s[0] * s[1] * s[2])]
    if case["kind"] == "batch":
        s = (case["n1"], case["n2"], case["n3"])
        return [(lv, "th", s, case["stride"], case["offset0"], s[0] * s[1] * s[2]) for lv in _levels(case)]
    if case["kind"] == "chain":
        return [(case["level"] - i, "th", s, h, o, D) for i, (o, h, D, s) in enumerate(_stages(case))]
    return []


def _rotations(algo, split, stride, offset0, D, slots):
    n1, n2, n3 = split
    if algo == "diag":
        r = [stride * t for t in range(1, D)] + [offset0]
    elif algo == "th":
        r = ([stride * i for i in range(1, n1)] + [stride * n1 * j for j in range(1, n2)]
             + [offset0 + stride * n1 * n2 * k for k in range(n3)])
    else:
        r = [stride * i for i in range(1, n1)] + [offset0 + stride * n1 * j for j in range(n2)]
    return {x % slots for x in r} - {0}


def _keys_needed(case):
    if case["kind"] == "rotation":
        return [case["rot"]]
    slots = synth.param_set(case["params"]).n // 2
    need = set()
    for _, algo, split, stride, offset0, D in _lts(case):
        need |= _rotations(algo, split, stride, offset0, D, slots)
    return sorted(need)


def _beta(ps, level):
    return -(-level // ps.alpha)


# ------------------------------------------------------------------ inputs, from the seed alone
def _uniform(seed, tag, moduli, n, count):
    """[count][len(moduli)][n] residues, row i uniform in [0, moduli[i])."""
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1000003 + synth.stream_id(tag)) % (1 << 62))
    out = torch.empty((count, len(moduli), n), dtype=torch.int64, device=DEV)
    i = 0
    while i < len(moduli):  # moduli of one width are drawn together, then brought into range
        j = i
        while j < len(moduli) and int(moduli[j]).bit_length() == int(moduli[i]).bit_length():
            j += 1
        w = int(moduli[i]).bit_length()
        out[:, i:j].random_(0, 1 << w, generator=g)
        q = torch.tensor([int(m) for m in moduli[i:j]], dtype=torch.int64, device=DEV)[:, None]
        out[:, i:j] -= torch.where(out[:, i:j] >= q, q, torch.zeros_like(q))
        i = j
    return out


def _key(ps, seed, r):
    beta_max = _beta(ps, ps.L)
    return _uniform(seed, f"key/{r}", ps.moduli, ps.n, 2 * beta_max).view(beta_max, 2, ps.L + ps.k, ps.n)


def _diags(ps, seed, i, D):
    return _uniform(seed, f"diags/{i}", ps.moduli, ps.n, D)


def _ct(ps, seed, i, level):
    return _uniform(seed, f"ct/{i}", ps.q[:level], ps.n, 2)


def _poly(ps, seed, level, ext):
    return _uniform(seed, "poly", list(ps.q[:level]) + (list(ps.p) if ext else []), ps.n, 1)[0]


# ------------------------------------------------------------------ what a program keeps, and one pass
class _State:
    def __init__(self, case):
        self.case = case
        self.ctx = binding.Context.from_params(synth.param_set(case["params"]))
        self.fs = []

    def __del__(self):
        try:
            torch.cuda.synchronize()
            for f in self.fs:
                f.free()
            self.ctx.close()
        except Exception:
            pass


def prepare(case, seed):
    ps = synth.param_set(case["params"])
    st = _State(case)
    g, kind = st.ctx, case["kind"]
    for r in _keys_needed(case):
        g.upload_rotation_key_device(r, _key(ps, seed, r))
    if kind in ("lt", "batch", "chain"):
        lts = _lts(case)
        for i, (_, _, _, stride, offset0, D) in enumerate(lts if kind == "chain" else lts[:1]):
            st.fs.append(g.upload_diagonals_device(_diags(ps, seed, i, D), stride=stride, level=ps.L,
                                                   offset0=offset0))
    level = case["level"]
    if kind == "batch":
        st.cts = [g.ct_wrap(_ct(ps, seed, i, lv), lv) for i, lv in enumerate(_levels(case))]
        st.outs = [g.ct_empty(c.level - 1) for c in st.cts]
    elif kind in ("lt", "chain"):
        st.ct = g.ct_wrap(_ct(ps, seed, 0, level), level)
        st.out = g.ct_empty(level - (len(st.fs) if kind == "chain" else 1))
    elif kind == "rotation":
        st.c = _ct(ps, seed, 0, level)
        st.digits = torch.empty((g.beta(level), level + ps.k, ps.n), dtype=torch.int64, device=DEV)
        st.x = torch.empty((2, level + ps.k, ps.n), dtype=torch.int64, device=DEV)
        st.y = torch.empty((2, level, ps.n), dtype=torch.int64, device=DEV)
    elif kind == "ntt":
        st.x = _poly(ps, seed, level, True)
        st.y = torch.empty((2,) + tuple(st.x.shape), dtype=torch.int64, device=DEV)
    else:
        st.x = _poly(ps, seed, level, case["op"] != "rescale")
        st.y = torch.empty((level if case["op"] == "moddown" else level - 1, ps.n), dtype=torch.int64, device=DEV)
    torch.cuda.synchronize()
    return st


def run(st):
    c, g = st.case, st.ctx
    kind, level = c["kind"], c["level"]
    if kind == "lt":
        split = (c["n1"], c["n2"], c["n3"])
        out, _ = g.lt_eval(st.ct, st.fs[0], c["algo"], split, out=st.out)
        return out.tensor
    if kind == "batch":
        n = c["count"]
        g.lt_eval_batch(st.cts, [st.fs[0]] * n, ["th"] * n, [(c["n1"], c["n2"], c["n3"])] * n, st.outs)
        return [o.tensor for o in st.outs]
    if kind == "chain":
        out, _ = g.lt_eval_chain(st.ct, st.fs, splits=[s for _, _, _, s in _stages(c)], out=st.out)
        return out.tensor
    if kind == "rotation":
        g.decompose(st.c[1], level, digits=st.digits)
        g.ks_inner(level, st.digits, c["rot"], c["rot"], x0=st.c[0], lift_x0=True, out0=st.x[0], out1=st.x[1])
        g.moddown(st.x[0], level, out=st.y[0])
        g.moddown(st.x[1], level, out=st.y[1])
        return [st.digits, st.y]
    if kind == "ntt":
        st.y[0].copy_(st.x)
        st.y[1].copy_(st.x)
        g.ntt(st.y[0], level, True, False)
        g.ntt(st.y[1], level, True, True)
        return st.y
    if c["op"] == "moddown":
        return g.moddown(st.x, level, out=st.y)
    if c["op"] == "moddown_rescale":
        return g.moddown_rescale(st.x, level, out=st.y)
    return g.rescale(st.x, level, out=st.y)


# ------------------------------------------------------------------ bytes and operations
def work(case):
    """Bytes: diagonals and keys at their information content (whole bytes of
    a residue, every needed one once), ciphertexts and polynomials at the 8
    bytes of the interface.  Operations: two per residue multiply-accumulate
    and per NTT butterfly, counted from the algorithm of the case."""
    ps = synth.param_set(case["params"])
    n, k = ps.n, ps.k
    width = lambda m: -(-int(m).bit_length() // 8)
    ext_b = lambda lv: sum(width(m) for m in list(ps.q[:lv]) + list(ps.p)) * n
    q_b = lambda lv: sum(width(m) for m in ps.q[:lv]) * n
    bf = n / 2 * ps.log_n
    dec = lambda lv: (lv + _beta(ps, lv) * (lv + k) - lv) * bf + _beta(ps, lv) * (lv + k) * ps.alpha * n
    down = lambda s, t: (s + t) * bf + s * t * n
    kind, lv = case["kind"], case["level"]
    by = ops = 0.0
    if kind in ("lt", "batch", "chain"):
        seen = set()
        slots = n // 2
        for i, (l, algo, split, stride, offset0, D) in enumerate(_lts(case)):
            n1, n2, n3 = split
            f = 0 if kind == "batch" else i
            if f not in seen:  # the first LT of a batch is its highest level
                by += D * (q_b(l) if algo == "bsgs" else ext_b(l))
                seen.add(f)
            rots = _rotations(algo, split, stride, offset0, D, slots)
            for r in rots:
                if ("key", r) not in seen:
                    by += 2 * _beta(ps, l) * ext_b(l)
                    seen.add(("key", r))
            by += 2 * l * n * 8 + 2 * (l - 1) * n * 8
            ext, b = l + k, _beta(ps, l)
            outer = sum(1 for j in range({"th": n3, "diag": 1}.get(algo, n2))
                        if (offset0 + stride * (D // {"th": n3, "diag": 1}.get(algo, n2)) * j) % slots)
            if algo == "bsgs":
                ops += 2 * D * l * n + len(rots) * (dec(l) + 2 * b * ext * n + 2 * down(k, l)) + 2 * down(1, l - 1)
                continue
            baby = n1 - 1 if algo == "th" and n2 > 1 else 0  # baby indices with a digit set of their own
            mid = n1 * (n2 - 1) if algo == "th" else (D - 1 if algo == "diag" else 0)
            inner = mid + outer + (n1 - 1 if algo != "diag" else 0)
            ops += 2 * D * ext * n + inner * 2 * b * ext * n
            ops += (1 + baby + outer) * dec(l) + (baby + outer) * down(k, l) + 2 * down(k + 1, l - 1)
    elif kind == "rotation":
        by = 2 * lv * n * 8 + 2 * _beta(ps, lv) * ext_b(lv) + (_beta(ps, lv) * (lv + k) + 2 * lv) * n * 8
        ops = dec(lv) + 2 * _beta(ps, lv) * (lv + k) * n + 2 * down(k, lv)
    elif kind == "ntt":
        by = 3 * (lv + k) * n * 8
        ops = 2 * (lv + k) * bf
    else:
        s, t = {"moddown": (k, lv), "moddown_rescale": (k + 1, lv - 1), "rescale": (1, lv - 1)}[case["op"]]
        by = (s + t + t) * n * 8
        ops = down(s, t)
    return {"bytes": float(by), "flops": 2.0 * ops}


# ------------------------------------------------------------------ the same outputs from the definitions
def _mul30(a, c, q):
    """a c mod q for 0 <= a < q < 2^60, 0 <= c < 2^30: the double quotient is
    within one of the true one and the wrapped 64-bit remainder is exact."""
    t = torch.floor(a.double() * c.double() / q.double()).long() if torch.is_tensor(c) else \
        torch.floor(a.double() * float(c) / q.double()).long()
    r = a * c - t * q
    r = torch.where(r < 0, r + q, r)
    return torch.where(r >= q, r - q, r)


def _mulmod(a, b, q):
    hi = _mul30(_mul30(a, b >> 30, q), 1 << 30, q)
    return _add(hi, _mul30(a, b & ((1 << 30) - 1), q), q)


def _add(a, b, q):
    s = a + b
    return torch.where(s >= q, s - q, s)


def _sub(a, b, q):
    s = a - b
    return torch.where(s < 0, s + q, s)


class _Ring:
    """R_q for a list of moduli; polynomials are [..., limb, N], NTT domain in bit-reversed order."""

    def __init__(self, ps):
        self.ps, self.n, self.log_n, self.k = ps, ps.n, ps.log_n, ps.k
        idx = torch.arange(self.n, device=DEV)
        self.brv = torch.zeros_like(idx)
        for b in range(self.log_n):
            self.brv |= ((idx >> b) & 1) << (self.log_n - 1 - b)
        self.tw = {}

    def basis(self, level, ext=True):
        return list(self.ps.q[:level]) + (list(self.ps.p) if ext else [])

    @staticmethod
    def q(mods):
        return torch.tensor([int(m) for m in mods], dtype=torch.int64, device=DEV)[:, None]

    def const(self, a, cs, mods):
        return _mulmod(a, self.q([int(c) % int(m) for c, m in zip(cs, mods)]).expand_as(a), self.q(mods))

    def twiddles(self, m):
        """psi^brv(i) and psi^-brv(i), psi = x^((m-1)/2N) for the smallest x with psi^N = -1."""
        if m not in self.tw:
            x = 2
            while pow(x, (m - 1) // 2, m) != m - 1:
                x += 1
            w = pow(x, (m - 1) // (2 * self.n), m)
            q = torch.tensor(m, dtype=torch.int64, device=DEV)
            out = []
            for base in (w, pow(w, -1, m)):
                t = torch.ones(1, dtype=torch.int64, device=DEV)
                while t.numel() < self.n:
                    step = torch.full_like(t, pow(base, t.numel(), m))
                    t = torch.cat([t, _mulmod(t, step, q)])
                out.append(t[self.brv])
            self.tw[m] = out
        return self.tw[m]

    def ntt(self, a, mods, inverse=False):
        shape, L = a.shape, len(mods)
        tw = torch.stack([self.twiddles(int(m))[1 if inverse else 0] for m in mods])
        q = self.q(mods)[:, :, None]
        a = a.reshape(-1, L, self.n)
        stages = [1 << s for s in range(self.log_n)]
        for m in reversed(stages) if inverse else stages:
            v = a.view(-1, L, m, 2, self.n // (2 * m))
            w = tw[:, m:2 * m, None].expand(L, m, self.n // (2 * m))
            x, y = v[..., 0, :], v[..., 1, :]
            if inverse:
                a = torch.stack([_add(x, y, q), _mulmod(_sub(x, y, q), w.expand_as(x), q)], dim=3)
            else:
                y = _mulmod(y, w.expand_as(y), q)
                a = torch.stack([_add(x, y, q), _sub(x, y, q)], dim=3)
            a = a.reshape(-1, L, self.n)
        a = a.reshape(shape)
        return self.const(a, [pow(self.n, -1, int(m)) for m in mods], mods) if inverse else a

    def auto(self, a, r):
        """phi_r: the evaluation point 2 brv(s) + 1 of word s moves to its 5^r-th power."""
        r %= self.n // 2
        if r == 0:
            return a
        e = (pow(5, r, 2 * self.n) * (2 * self.brv + 1)) % (2 * self.n)
        return a[..., self.brv[(e - 1) // 2]]

    def convert(self, x, src, dst):
        """Fast basis conversion of NTT-domain limbs: sum_j [x_j (S/s_j)^-1]_{s_j} [S/s_j]_t, as NTT-domain limbs."""
        S = math.prod(int(s) for s in src)
        y = self.ntt(x, src, True)
        y = self.const(y, [pow(S // int(s) % int(s), -1, int(s)) for s in src], src)
        q = self.q(dst)
        out = torch.zeros(x.shape[:-2] + (len(dst), self.n), dtype=torch.int64, device=DEV)
        for j, s in enumerate(src):
            yj = (y[..., j:j + 1, :].expand_as(out)) % q
            out = _add(out, self.const(yj, [S // int(s)] * len(dst), dst), q)
        return self.ntt(out, dst)

    def decompose(self, c, level):
        basis, out = self.basis(level), []
        for b in range(_beta(self.ps, level)):
            own = list(range(b * self.ps.alpha, min(level, (b + 1) * self.ps.alpha)))
            rest = [t for t in range(len(basis)) if t not in own]
            d = torch.empty(c.shape[:-2] + (len(basis), self.n), dtype=torch.int64, device=DEV)
            d[..., own, :] = c[..., own, :]
            d[..., rest, :] = self.convert(c[..., own, :], [basis[j] for j in own], [basis[t] for t in rest])
            out.append(d)
        return out

    def down(self, x, src_rows, src, dst):
        S = math.prod(int(s) for s in src)
        conv = self.convert(x[..., src_rows, :], src, dst)
        return self.const(_sub(x[..., :len(dst), :], conv, self.q(dst)), [pow(S % int(m), -1, int(m)) for m in dst],
                          dst)

    def moddown(self, x, level):
        return self.down(x, list(range(level, level + self.k)), self.ps.p, self.basis(level, False))

    def moddown_rescale(self, x, level):
        return self.down(x, list(range(level - 1, level + self.k)), [self.ps.q[level - 1]] + list(self.ps.p),
                         self.basis(level - 1, False))

    def rescale(self, x, level):
        return self.down(x, [level - 1], [self.ps.q[level - 1]], self.basis(level - 1, False))

    def lift(self, c, level):
        P = math.prod(int(p) for p in self.ps.p)
        q = self.basis(level, False)
        return torch.cat([self.const(c, [P] * level, q), torch.zeros(c.shape[:-2] + (self.k, self.n),
                                                                    dtype=torch.int64, device=DEV)], dim=-2)

    def inner(self, digits, key, level):
        rows = list(range(level)) + list(range(self.ps.L, self.ps.L + self.k))
        q = self.q(self.basis(level))
        acc = [torch.zeros_like(digits[0]) for _ in range(2)]
        for b, d in enumerate(digits):
            for c in range(2):
                acc[c] = _add(acc[c], _mulmod(d, key[b, c, rows].expand_as(d), q), q)
        return acc

    def hoisted(self, x0, digits, key, r, level):
        """(phi_r(x0) + <phi_r(d), swk_0>, <phi_r(d), swk_1>)"""
        acc = self.inner([self.auto(d, r) for d in digits], key, level)
        return _add(self.auto(x0, r), acc[0], self.q(self.basis(level))), acc[1]


def _exact_lt(R, c0, c1, f, keys, level, algo, split, stride, offset0):
    """One LT of c0, c1 ([..., level, N]) by the definition of its algorithm; f [D][L + k][N]."""
    n1, n2, n3 = split
    D, bs = n1 * n2 * n3, algo == "bsgs"
    if algo == "dh":
        n3, n2 = n2, 1
    rows = list(range(level)) + ([] if bs else list(range(R.ps.L, R.ps.L + R.k)))
    basis = R.basis(level, not bs)
    q, slots = R.q(basis), R.n // 2
    per = D // (n2 if bs else n3)  # diagonals per outer index
    outer = [(offset0 + stride * per * k) % slots for k in range(D // per)]
    U = [[torch.zeros(c0.shape[:-2] + (len(basis), R.n), dtype=torch.int64, device=DEV) for _ in range(2)]
         for _ in outer]

    def rotate_bsgs(x0, x1, r):
        t = R.inner(R.decompose(R.auto(x1, r), level), keys(r), level)
        return _add(R.auto(x0, r), R.moddown(t[0], level), q), R.moddown(t[1], level)

    def use(t, a, b):
        for k, r in enumerate(outer):
            fh = R.auto(f[per * k + t][rows], -r).expand_as(a)
            U[k][0] = _add(U[k][0], _mulmod(a, fh, q), q)
            U[k][1] = _add(U[k][1], _mulmod(b, fh, q), q)

    if bs:
        use(0, c0, c1)
        for i in range(1, n1):
            use(i, *rotate_bsgs(c0, c1, stride * i % slots))
    else:
        d0 = R.decompose(c1, level)
        for i in range(n1):
            if i == 0:
                a, b, d = R.lift(c0, level), R.lift(c1, level), d0
            else:
                a, b = R.hoisted(R.lift(c0, level), d0, keys(stride * i % slots), stride * i, level)
                d = R.decompose(R.moddown(b, level), level) if n2 > 1 else None
            use(i, a, b)
            for j in range(1, n2):
                r = stride * n1 * j % slots
                use(n1 * j + i, *R.hoisted(a, d, keys(r), r, level))
    acc = [torch.zeros_like(U[0][0]) for _ in range(2)]
    for (u0, u1), r in zip(U, outer):
        if r and bs:
            u0, u1 = rotate_bsgs(u0, u1, r)
        elif r:
            u0, u1 = R.hoisted(u0, R.decompose(R.moddown(u1, level), level), keys(r), r, level)
        acc = [_add(acc[0], u0, q), _add(acc[1], u1, q)]
    fin = R.rescale if bs else R.moddown_rescale
    return fin(acc[0], level), fin(acc[1], level)


def exact(case, seed):
    ps = synth.param_set(case["params"])
    R, kind, level = _Ring(ps), case["kind"], case["level"]
    keys = lambda r: _key(ps, seed, r)
    if kind == "lt":
        (lv, algo, split, stride, offset0, D), = _lts(case)
        c = _ct(ps, seed, 0, lv)
        return torch.stack(_exact_lt(R, c[0], c[1], _diags(ps, seed, 0, D), keys, lv, algo, split, stride, offset0))
    if kind == "chain":
        c = _ct(ps, seed, 0, level)
        for i, (lv, algo, split, stride, offset0, D) in enumerate(_lts(case)):
            c = torch.stack(_exact_lt(R, c[0], c[1], _diags(ps, seed, i, D), keys, lv, algo, split, stride, offset0))
        return c
    if kind == "batch":
        lts = _lts(case)
        f = _diags(ps, seed, 0, lts[0][5])
        out = [None] * len(lts)
        for lv in set(_levels(case)):  # the ciphertexts of one level together
            at = [i for i, l in enumerate(_levels(case)) if l == lv]
            c = torch.stack([_ct(ps, seed, i, lv) for i in at])
            _, algo, split, stride, offset0, _ = lts[at[0]]
            o0, o1 = _exact_lt(R, c[:, 0], c[:, 1], f, keys, lv, algo, split, stride, offset0)
            for p, i in enumerate(at):
                out[i] = torch.stack([o0[p], o1[p]])
        return out
    if kind == "rotation":
        c = _ct(ps, seed, 0, level)
        d = R.decompose(c[1], level)
        x0, x1 = R.hoisted(R.lift(c[0], level), d, keys(case["rot"]), case["rot"], level)
        return [torch.stack(d), torch.stack([R.moddown(x0, level), R.moddown(x1, level)])]
    if kind == "ntt":
        x, basis = _poly(ps, seed, level, True), R.basis(level)
        return torch.stack([R.ntt(x, basis), R.ntt(x, basis, True)])
    x = _poly(ps, seed, level, case["op"] != "rescale")
    return {"moddown": R.moddown, "moddown_rescale": R.moddown_rescale, "rescale": R.rescale}[case["op"]](x, level)
