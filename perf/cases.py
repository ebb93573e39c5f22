"""The workloads that the library's speed is measured on: calls that a user's
program makes through the public entry points (Plan.contract, Plan.backward, contract
with autograd, Plan.contract_complex), over the sizes, forms and directions of the
method's own uses.  The alignment transforms are part of every contraction;
Plan.align, which runs one alone, is a means of checking and not listed.

A case names its contraction by the einsum string, the moduli, the block size
of each letter ("a=32 b=32 ..."), the charge signs of the two operands and the
precision form.  Optional: sector counts below the group order ("b=4 d=2",
coefficient +-G/H) and `ragged` (sector sizes between half and the whole of the
block size, in padded blocks).  `op`:

  contract          w = einsum(u, v)
  grad              w and the gradients of u and v for an upstream gradient of w (Plan.backward)
  loss              y = einsum(u, v), loss = sum(y * y), gradients of u and v through autograd
  transfer          X = E.A, E' = X.A (two contractions, "ab,asg->bsg" and "bsg,bsd->gd")
  transfer_complex  the same for complex A, E' = X.conj(A)
"""
import itertools
import math

import torch

import paper_2007_08056_gb300 as sc

STEP1, STEP2 = "ab,asg->bsg", "bsg,bsd->gd"


def _ladder(G, virt, occ, form, op="contract"):
    return {"op": op, "form": form, "einsum": "abcd,cdij->abij", "moduli": str(G),
            "dims": "a=%d b=%d c=%d d=%d i=%d j=%d" % (virt, virt, virt, virt, occ, occ),
            "su": "++--", "sv": "++--"}


def _transfer(G, bond, phys, form, op="transfer"):
    return {"op": op, "form": form, "einsum": STEP1, "moduli": str(G),
            "dims": "a=%d b=%d s=%d g=%d" % (bond, bond, phys, bond), "su": "+-", "sv": "++-"}


def _peps(moduli, virt, phys, form):
    return {"op": "loss", "form": form, "einsum": "uldrp,uldr->p", "moduli": moduli,
            "dims": "u=%d l=%d d=%d r=%d p=%d" % (virt, virt, virt, virt, phys),
            "su": "++--+", "sv": "--++"}


def _generic(s, t, v, G, dims, form, op="contract"):
    """s free modes of u, t free modes of v, v contracted modes."""
    fu, c, fv = "abc"[:s], "klm"[:v], "xyz"[:t]
    return {"op": op, "form": form, "einsum": "%s%s,%s%s->%s%s" % (fu, c, c, fv, fu, fv),
            "moduli": str(G), "dims": " ".join("%s=%d" % (x, d) for x, d in zip(fu + c + fv, dims)),
            "su": "+" * s + "-" * v, "sv": "+" * v + "-" * t}


def _padded(G, virt, occ, form):
    """The ladder with sub-group modes (G/2 and 2 sectors) and sectors of unequal size."""
    return dict(_ladder(G, virt, occ, form), sectors="b=%d d=2 j=%d" % (max(1, G // 2), max(1, G // 2)),
                ragged=True)


def listed():
    n = lambda name, c: dict(c, name=name)
    return [
        # the method's own example (order 4, Z_3, blocks of 4): one small contraction, as
        # they occur by the thousand inside a larger tensor-network program; latency counts
        n("order4_split", _ladder(3, 4, 4, "split_bf16")),
        n("order4_fp64", _ladder(3, 4, 4, "fp64")),
        # one site of an MPS sweep, bond 8 x 128, physical 8 x 2: two chained contractions
        n("transfer_split", _transfer(8, 128, 2, "split_bf16")),
        n("transfer_fp64", _transfer(8, 128, 2, "fp64")),
        # the same for complex tensors (time evolution), with conj(A)
        n("transfer_complex_split", _transfer(8, 128, 2, "split_bf16", "transfer_complex")),
        # coupled-cluster particle-particle ladder, virtual 8 x 32, occupied 8 x 8: the largest
        n("ladder_split", _ladder(8, 32, 8, "split_bf16")),
        n("ladder_tf32", _ladder(8, 32, 8, "tf32")),
        # the ladder with many small sectors, forward and backward (amplitude optimisation)
        n("ladder16_split_grad", _ladder(16, 16, 4, "split_bf16", "grad")),
        # gradient of a PEPS tensor and its environment under Z_2 x Z_3: bound by memory
        n("peps_loss_fp64", _peps("2,3", 16, 2, "fp64")),
        # odd sector size 23: no row is a multiple of any tile or load width
        n("odd_split", _generic(2, 2, 2, 4, (23,) * 6, "split_bf16")),
        # a tall operand against a small one (PEPS boundary): 40960 x 640 x 640 for each irrep
        n("tall_split", {"op": "contract", "form": "split_bf16", "einsum": "ijkl,klmn->ijmn", "moduli": "10",
                         "dims": "i=64 j=64 k=8 l=8 m=8 n=8", "su": "++--", "sv": "++--"}),
        # sub-group modes and sectors of unequal size in padded blocks
        n("padded_split", _padded(8, 24, 8, "split_bf16")),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# The most that a drawn case costs (each below the largest listed one): flops in the
# tensor-core forms and in float64 (for sub-group modes and padded sectors, those of the
# aligned product with all its absent rows and columns), bytes of operands and results.
MOST = {"split_bf16": 300e9, "tf32": 300e9, "fp64": 4e9}
MOST_BYTES = 2.5e9


def draw(rng):
    while True:
        family = rng.choice(["small", "transfer", "ladder", "peps", "generic", "padded"])
        form = rng.choice(["split_bf16", "split_bf16", "tf32", "fp64"])
        G = rng.randint(2, 16)
        if family == "small":
            c = _ladder(rng.randint(2, 6), rng.randint(2, 8), rng.randint(2, 8), form,
                        rng.choice(["contract", "grad"]))
        elif family == "transfer":
            c = _transfer(G, _log(rng, 16, 160), rng.randint(1, 4), form,
                          rng.choice(["transfer", "transfer", "transfer_complex"]))
        elif family == "ladder":
            c = _ladder(G, _log(rng, 6, 40), _log(rng, 2, 16), form, rng.choice(["contract", "grad"]))
        elif family == "peps":
            c = _peps(rng.choice(["2,3", "2", "3", "5"]), rng.randint(4, 17), rng.randint(1, 3),
                      rng.choice(["fp64", "split_bf16"]))
        elif family == "generic":
            s, t, v = rng.choice([1, 2, 3]), rng.choice([1, 2, 3]), rng.choice([1, 2])
            c = _generic(s, t, v, rng.randint(2, 8), [_log(rng, 3, 90) for _ in range(s + t + v)], form,
                         rng.choice(["contract", "contract", "grad"]))
        else:
            c = _padded(rng.choice([4, 6, 8, 12]), rng.randint(6, 24), rng.randint(3, 10), form)
        w = work(c)
        if (max(w["flops"], _aligned(c)) <= MOST[form] and w["bytes"] <= MOST_BYTES
                and _stored(c) * 8 <= 2 * MOST_BYTES):
            return c


# ---------------------------------------------------------------- the case's tensors

def _map(text):
    return {p.split("=")[0]: int(p.split("=")[1]) for p in text.split()}


class _Law:
    """One tensor: its letters, block sizes, sector counts and sizes, signs and the group."""

    def __init__(self, case, labels, signs):
        self.moduli = tuple(int(m) for m in str(case["moduli"]).split(","))
        G = math.prod(self.moduli)
        dims, sect = _map(case["dims"]), _map(case.get("sectors", ""))
        dims.setdefault("d", dims.get("g", 0))      # the second leg of a transfer step
        self.labels, self.signs = labels, tuple(1 if s == "+" else -1 for s in signs)
        self.dims = tuple(dims[x] for x in labels)
        self.sectors = tuple(sect.get(x, G) for x in labels)
        self.sizes = None
        if case.get("ragged"):
            self.sizes = tuple(tuple(d - (7 * ord(x) + 5 * q) % (d // 2 + 1) for q in range(h))
                               for x, d, h in zip(labels, self.dims, self.sectors))
        self.general = "sectors" in case or self.sizes is not None
        self.shape = self.sectors[:-1] + self.dims

    def spec(self, negate=False):
        signs, charge = tuple(-s for s in self.signs) if negate else self.signs, (0,) * len(self.moduli)
        return (signs, charge, self.dims) + ((self.sectors, self.sizes) if self.general else ())

    def charge(self, k, q):
        """Charge that sector q of mode k carries, one component for each modulus."""
        if len(self.moduli) == 1:
            return (self.signs[k] * (self.moduli[0] // self.sectors[k]) * q % self.moduli[0],)
        out = []
        for m in reversed(self.moduli):
            out.append(self.signs[k] * (q % m) % m)
            q //= m
        return tuple(reversed(out))

    def total(self, modes, sectors):
        c = [self.charge(k, q) for k, q in zip(modes, sectors)]
        return tuple(sum(x[i] for x in c) % m for i, m in enumerate(self.moduli))

    def size(self, k, q):
        return self.dims[k] if self.sizes is None else self.sizes[k][q]

    def blocks(self):
        """Sectors of every block that the conservation law allows."""
        last = len(self.labels) - 1
        of = {}
        for q in range(self.sectors[last]):
            of[self.total([last], [q])] = q
        for qs in itertools.product(*(range(h) for h in self.sectors[:-1])):
            t = self.total(range(last), qs)
            q = of.get(tuple(-x % m for x, m in zip(t, self.moduli)))
            if q is not None:
                yield qs + (q,)

    def lengths(self, modes):
        """{charge: number of index values of these modes that carry it}."""
        out = {(0,) * len(self.moduli): 1}
        for k in modes:
            new = {}
            for t, n in out.items():
                for q in range(self.sectors[k]):
                    u = tuple((x + y) % m for x, y, m in zip(t, self.charge(k, q), self.moduli))
                    new[u] = new.get(u, 0) + n * self.size(k, q)
            out = new
        return out


def _laws(case):
    ins, out = case["einsum"].split("->")
    lu, lv = ins.split(",")
    U, V = _Law(case, lu, case["su"]), _Law(case, lv, case["sv"])
    return U, V, _out_law(case, U, V, out)


def _out_law(case, U, V, out):
    # contracted modes carry opposite signs in u and v (sigma = -1) or equal ones (+1)
    shared = [x for x in U.labels if x in V.labels]
    sigma = U.signs[U.labels.index(shared[0])] * V.signs[V.labels.index(shared[0])] if shared else -1
    sign = lambda x: U.signs[U.labels.index(x)] if x in U.labels else -sigma * V.signs[V.labels.index(x)]
    return _Law(case, out, "".join("+" if sign(x) > 0 else "-" for x in out))


def _second(case, X):
    """Laws of the second contraction of a transfer step, whose u is X and whose result is E'."""
    A = _Law(case, "bsd", case["sv"])
    return A, _out_law(case, X, A, "gd")


def _counts(U, V):
    """(flops, entries of u and of v that take part) of one contraction."""
    pos = lambda law, keep: [k for k, x in enumerate(law.labels) if keep(x)]
    shared = lambda x: x in U.labels and x in V.labels
    neg = lambda q, m: tuple(-x % y for x, y in zip(q, m))
    fu, c = U.lengths(pos(U, lambda x: not shared(x))), U.lengths(pos(U, shared))
    fv = V.lengths(pos(V, lambda x: not shared(x)))
    k0 = pos(U, shared)
    flip = bool(k0) and U.signs[k0[0]] == V.signs[V.labels.index(U.labels[k0[0]])]
    flops = nu = nv = 0
    for q, k in c.items():
        m = fu.get(neg(q, U.moduli), 0)
        n = fv.get(neg(q, U.moduli) if flip else q, 0)
        if m and n:
            flops, nu, nv = flops + 2 * m * n * k, nu + m * k, nv + n * k
    return flops, nu, nv


def _entries(law):
    return law.lengths(range(len(law.labels))).get((0,) * len(law.moduli), 0) if law.labels else 1


def _stored(case):
    U, V, W = _laws(case)
    return sum(math.prod(t.shape) for t in (U, V, W)) * (2 if case["op"] in ("grad", "loss") else 1)


def _aligned(case):
    """Flops of the aligned product with every explicit sector and whole blocks."""
    U, V, _ = _laws(case)
    out = 2.0 * math.prod(U.moduli)
    for modes in ([(x, h, d) for x, h, d in zip(U.labels, U.sectors, U.dims) if x not in V.labels],
                  [(x, h, d) for x, h, d in zip(U.labels, U.sectors, U.dims) if x in V.labels],
                  [(x, h, d) for x, h, d in zip(V.labels, V.sectors, V.dims) if x not in U.labels]):
        out *= math.prod(h for _, h, _ in modes[:-1]) * math.prod(d for _, _, d in modes)
    return out


def work(case):
    """What one pass cannot do without: the entries that take part read once, results
    written once, the symmetry-reduced multiply-adds (four real ones for a complex one)."""
    U, V, W = _laws(case)
    f, nu, nv = _counts(U, V)
    nw = _entries(W)
    if case["op"].startswith("transfer"):
        A2, E2 = _second(case, W)
        f2, _, _ = _counts(W, A2)
        cplx = case["op"] == "transfer_complex"
        return {"bytes": (16 if cplx else 8) * (nu + nv + _entries(E2)), "flops": (4 if cplx else 1) * (f + f2)}
    if case["op"] == "contract":
        return {"bytes": 8 * (nu + nv + nw), "flops": f}
    # u, v (and the upstream gradient) read, w and the whole gradients written
    return {"bytes": 8 * (nu + nv + 2 * nw + _entries(U) + _entries(V)), "flops": 3 * f}


# ---------------------------------------------------------------- a user's program

def _normal(shape, seed, scale, complex_=False):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda",
                       dtype=torch.complex128 if complex_ else torch.float64) * scale


def _inputs(case, seed):
    U, V, W = _laws(case)
    cplx = case["op"] == "transfer_complex"
    k = math.prod(h * d for x, d, h in zip(U.labels, U.dims, U.sectors) if x in V.labels)
    x = {"u": _normal(U.shape, 3 * seed + 1, 1.0 / math.sqrt(k), cplx), "v": _normal(V.shape, 3 * seed + 2, 1.0, cplx)}
    if case["op"] == "grad":
        x["gw"] = _normal(W.shape, 3 * seed + 3, 1.0)
    for law, name in ((U, "u"), (V, "v"), (W, "gw")):
        if law.sizes is not None and name in x:
            x[name] = x[name] * _mask(law)      # padding holds zeros
    return x


def prepare(case, seed):
    U, V, W = _laws(case)
    s = dict(_inputs(case, seed), op=case["op"])
    s["plan"] = sc.Plan(case["einsum"], U.moduli, U.spec(), V.spec(), case["form"])
    if case["op"].startswith("transfer"):
        A2, _ = _second(case, W)
        s["plan2"] = sc.Plan(STEP2, U.moduli, s["plan"].sym_w, A2.spec(negate=case["op"] == "transfer_complex"),
                             case["form"])
    if case["op"] == "loss":
        s["u"].requires_grad_(True)
        s["v"].requires_grad_(True)
    return s


def run(s):
    op, u, v = s["op"], s["u"], s["v"]
    if op == "contract":
        return s["plan"].contract(u, v)
    if op == "transfer":
        return s["plan2"].contract(s["plan"].contract(u, v), v)
    if op == "transfer_complex":
        return s["plan2"].contract_complex(s["plan"].contract_complex(u, v), v, conj_v=True)
    if op == "grad":
        w = s["plan"].contract(u, v)
        gu, gv = s["plan"].backward(s["gw"], u, v)
        return {"w": w, "gu": gu, "gv": gv}
    y = sc.contract(s["plan"], u, v)
    gu, gv = torch.autograd.grad((y * y).sum(), (u, v))
    return {"w": y.detach(), "gu": gu, "gv": gv}


# Relative error (2-norm) of each form against float64 sums in another order, times about
# four: float64 up to 4e-15, and 1e-14 for `loss`, whose few outputs are sums of up to 14
# million terms of either sign; the split form 0.4e-11 to 2.5e-11 (it keeps 39 bits of each
# row's largest entry); TF32 2.9e-4 to 4.2e-4.
TOLERANCE = {"fp64": {"rel": 1.6e-14, "max": 2e-13}, "split_bf16": {"rel": 1e-10, "max": 1e-9},
             "tf32": {"rel": 1.7e-3, "max": 2e-2}}


def tolerance(case):
    if case["op"] == "loss":
        return {"rel": 6e-14, "max": 1e-12}
    return TOLERANCE[case["form"]]


# ---------------------------------------------------------------- the same in plain torch

def _mask(law):
    m = torch.zeros(law.shape, dtype=torch.float64, device="cuda")
    for q in law.blocks():
        m[q[:-1]][tuple(slice(0, law.size(k, x)) for k, x in enumerate(q))] = 1.0
    return m


def _contract(U, u, V, v, W):
    """Float64 contraction block by block: for each charge of the contracted modes, the
    blocks of u and v side by side in one matrix each, and one matrix product."""
    shared = [x for x in U.labels if x in V.labels]

    def matrices(law, t):
        free = [k for k, x in enumerate(law.labels) if x not in shared]
        con = [law.labels.index(x) for x in shared]
        rows = math.prod(law.dims[k] for k in free)
        got = {}
        for q in law.blocks():
            cq = tuple(q[k] for k in con)
            charge = U.total([U.labels.index(x) for x in shared], cq)
            block = t[q[:-1]].permute(free + con).reshape(rows, -1)
            got.setdefault(charge, {})[(tuple(q[k] for k in free), cq)] = block
        return got

    a, b = matrices(U, u), matrices(V, v)
    w = torch.zeros(W.shape, dtype=u.dtype, device="cuda")
    fu, fv = [x for x in U.labels if x not in shared], [x for x in V.labels if x not in shared]
    back = [(fu + fv).index(x) for x in W.labels]
    block_shape = [d for law, f in ((U, fu), (V, fv)) for x, d in zip(law.labels, law.dims) if x in f]
    for charge in sorted(set(a) & set(b)):
        cols = sorted({c for _, c in a[charge]} & {c for _, c in b[charge]})
        if not cols:
            continue

        def whole(m):
            keys = sorted({r for r, _ in m})
            zero = torch.zeros_like(next(iter(m.values())))
            return keys, torch.cat([torch.cat([m.get((r, c), zero) for c in cols], 1) for r in keys], 0)

        (ra, ma), (rb, mb) = whole(a[charge]), whole(b[charge])
        p = (ma @ mb.T).reshape(len(ra), ma.shape[0] // len(ra), len(rb), mb.shape[0] // len(rb))
        for i, x in enumerate(ra):
            for j, y in enumerate(rb):
                q = [(x + y)[k] for k in back]
                w[tuple(q[:-1])] += p[i, :, j, :].reshape(block_shape).permute(back)
    return w


def exact(case, seed):
    U, V, W = _laws(case)
    x = _inputs(case, seed)
    u, v = x["u"], x["v"]
    w = _contract(U, u, V, v, W)
    if case["op"] == "contract":
        return w
    if case["op"].startswith("transfer"):
        A2, E2 = _second(case, W)
        return _contract(W, w, A2, v.conj().resolve_conj() if case["op"] == "transfer_complex" else v, E2)
    gw = x["gw"] if case["op"] == "grad" else 2 * w
    return {"w": w, "gu": _contract(W, gw, V, v, U), "gv": _contract(U, u, W, gw, V)}
