"""Performance cases of the correlator library: what a user's program asks of it.

A program of this library makes one plan per operator, then evaluates it on the
propagators of many gauge configurations.  The cases take the library's operators
through its public evaluation calls (device buffers, host buffers, batches, sink
momentum, per-site values, the hadron-block form), in its three arithmetics and its
three algorithms, on lattices of the benchmark's sizes and on odd ones.

``exact`` evaluates the same sums in complex double with plain torch: the determinant
form by Laplace expansion along columns, and the projected block form by the explicit
sum over the assignments of source quarks to sink baryons.
"""
import itertools
import math

import torch

from paper_2201_04269_gb300 import Context, abi

OPS = ("proton", "dinucleon_I", "he3_I", "he3_II_s")
KAPPA = 0.5          # decay of the propagators in time, as in the benchmark
NOISE = 1e-3         # spread of the sites around a common slice value (noisy workload)

# Arithmetic one sink site cannot do without, in flops (8 per complex multiply-add, 4 with
# a real weight): the staged minor plan of the operator, the factor tree with its
# minors, and the direct sweep's determinants.
FLOPS = {
    ("egraph", "proton"): 2.916e4, ("egraph", "dinucleon_I"): 3.387e6, ("egraph", "he3_I"): 1.305e7,
    ("egraph", "he3_II_s"): 3.405e7, ("egraph", "he3_II"): 0.0, ("egraph", "dinucleon_II"): 0.0,
    ("tree", "proton"): 3.751e4, ("tree", "dinucleon_I"): 9.951e6, ("tree", "he3_I"): 6.382e7,
    ("direct", "proton"): 4.838e4,
}
# the block form: per sink site (projected blocks) and per tree evaluation
BLOCK_FLOPS = {"proton": (2.966e4, 3.36e2), "dinucleon_I": (3.318e5, 1.728e5), "he3_I": (3.954e5, 3.153e7),
               "he3_II_s": (4.873e5, 9.994e7)}


def listed():
    return [
        # the smallest production call: single-baryon correlator of one configuration on a 4^3 x 8 test lattice
        _case("proton_fp32_4x8", op="proton", prec="fp32", T=8, V3=64),
        # two-baryon correlator over eight time slices of 16^3 (the mid-size lattice of the benchmark)
        _case("dinucleon_fp32_16x8", op="dinucleon_I", prec="fp32", T=8, V3=4096),
        # three-baryon correlator with per-site values kept (site guard), odd spatial volume
        _case("he3_I_fp32_sites_11x3", op="he3_I", prec="fp32", T=3, V3=1331, sites=True),
        # the benchmark's headline operator and lattice, two time slices of 24^3
        _case("he3_II_s_fp32_24x2", op="he3_II_s", prec="fp32", T=2, V3=13824),
        # the same operator at nonzero sink momentum in double-float, two sets, odd lattice
        _case("he3_II_s_mixed_mom_9x2", op="he3_II_s", prec="mixed", sets=2, T=2, V3=729, px=1, py=-1, pz=2),
        # the full-precision reference evaluation of one small slice
        _case("he3_II_s_fp64_9x1", op="he3_II_s", prec="fp64", V3=729),
        # the factor-tree algorithm in double-float
        _case("he3_I_tree_mixed_8x1", path="tree", op="he3_I", prec="mixed", V3=512),
        # the direct index-set sweep in double, as a user checks a single-baryon plan
        _case("proton_direct_fp64_4x8", path="direct", op="proton", prec="fp64", T=8, V3=64),
        # all five operators of a configuration on two propagator sets of different lattices, one batched call
        _case("batch_fp32_8x4_6x3", path="batch", op="proton,dinucleon_I,dinucleon_II,he3_I,he3_II", prec="fp32",
              T=4, V3=512, T2=3, V3_2=216),
        # end to end from pinned host memory
        _case("dinucleon_fp32_host_16x4", path="host", op="dinucleon_I", prec="fp32", T=4, V3=4096),
        # hadron-block form, every sink baryon projected to a momentum, double-float
        _case("blocks_he3_II_s_mixed_16x4", path="blocks", op="he3_II_s", prec="mixed", T=4, V3=4096, px=0, py=1, pz=-1),
        # hadron-block form at a local sink in double
        _case("blocks_local_dinucleon_fp64_16x1", path="blocks_local", op="dinucleon_I", prec="fp64", V3=4096),
    ]


def draw(rng):
    """One more case of the listed ones' ranges."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def lattice(most, cubic):
        sites = log(64, most)
        T = rng.randint(1, min(8, max(1, sites // 32)))
        V3 = max(1, sites // T)
        return T, (max(2, int(round(V3 ** (1 / 3) - 0.3))) ** 3 if cubic else V3)

    kind = rng.choice(("fp32", "fp32", "fp32", "mixed", "mixed", "fp64", "tree", "direct", "batch", "host", "blocks",
                       "blocks_local"))
    noise = rng.choice((0.0, 0.0, NOISE))
    if kind in ("fp32", "mixed", "fp64"):
        op = rng.choice(OPS)
        most = {"fp32": (65536, 40000, 12000, 12000), "mixed": (65536, 16000, 6000, 4000),
                "fp64": (65536, 12000, 3000, 1200)}[kind][OPS.index(op)]
        mom = rng.random() < 0.3
        T, V3 = lattice(most, mom)
        p = [rng.randint(-2, 2) if mom else 0 for _ in range(3)]
        return _case(None, op=op, prec=kind, sets=rng.choice((1, 1, 2)) if T * V3 * 2 <= most else 1, T=T, V3=V3,
                     px=p[0], py=p[1], pz=p[2], sites=rng.random() < 0.3, noise=noise)
    if kind == "tree":
        op = rng.choice(OPS[:3])
        T, V3 = lattice({"proton": 32768, "dinucleon_I": 4000, "he3_I": 600}[op], False)
        return _case(None, path="tree", op=op, prec=rng.choice(("mixed", "fp64")), T=T, V3=V3, noise=noise)
    if kind == "direct":
        T, V3 = lattice(32768, False)
        return _case(None, path="direct", op="proton", prec=rng.choice(("mixed", "fp64")), T=T, V3=V3, noise=noise)
    if kind == "batch":
        T, V3 = lattice(3000, False)
        T2, V3_2 = lattice(1500, False)
        return _case(None, path="batch", op="proton,dinucleon_I,dinucleon_II,he3_I,he3_II",
                     prec=rng.choice(("fp32", "fp32", "mixed")), T=T, V3=V3, T2=T2, V3_2=V3_2, noise=noise)
    if kind == "host":
        op = rng.choice(OPS)
        T, V3 = lattice((32768, 20000, 8000, 8000)[OPS.index(op)], False)
        return _case(None, path="host", op=op, prec="fp32", T=T, V3=V3, noise=noise)
    if kind == "blocks":
        op = rng.choice(OPS)
        T, V3 = lattice(32768, True)
        return _case(None, path="blocks", op=op, prec=rng.choice(("mixed", "fp64")), T=T, V3=V3,
                     px=rng.randint(-1, 1), py=rng.randint(-1, 1), pz=rng.randint(-1, 1), noise=noise)
    T, V3 = lattice(16000, False)
    return _case(None, path="blocks_local", op=rng.choice(("proton", "dinucleon_I")), prec="fp64", T=T, V3=V3,
                 noise=noise)


def _case(name, path="egraph", op="", prec="", sets=1, T=1, V3=1, px=0, py=0, pz=0, sites=False, noise=0.0, T2=0,
          V3_2=0):
    c = dict(path=path, op=op, prec=prec, sets=sets, T=T, V3=V3, px=px, py=py, pz=pz, sites=sites, noise=noise, T2=T2,
             V3_2=V3_2)
    return dict(c, name=name) if name else c


# ----------------------------------------------------------------------------- inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _fields(case, seed):
    """Up and down propagators of every geometry of the case: complex Gaussian entries decaying
    in time, or (noisy) scattered around one matrix per slice."""
    out = []
    for g, (sets, T, V3) in enumerate(_geometries(case)):
        gen = torch.Generator(device=_device()).manual_seed(int(seed) * 16 + g)
        pair = []
        for _ in range(2):
            shape = (sets, T, V3, 12, 12)
            f = torch.randn(shape, dtype=torch.complex128, device=_device(), generator=gen)
            if case["noise"]:
                base = torch.randn((sets, T, 1, 12, 12), dtype=torch.complex128, device=_device(), generator=gen)
                f = base + case["noise"] * f
            decay = torch.exp(-KAPPA * torch.arange(T, dtype=torch.float64, device=_device()))
            pair.append((f * decay.view(1, T, 1, 1, 1)).contiguous())
        out.append(tuple(pair))
    return out


def _geometries(case):
    g = [(case["sets"], case["T"], case["V3"])]
    if case["path"] == "batch":
        g.append((1, case["T2"], case["V3_2"]))
    return g


def _momentum(case):
    p = (case["px"], case["py"], case["pz"])
    return p if any(p) else None


def _extent(V3):
    return int(round(V3 ** (1 / 3)))


class _State:
    """The context, the plans and the fields that a user's program keeps between calls."""

    def __init__(self, case, seed):
        self.case = case
        self.ctx = Context(0)
        self.fields = _fields(case, seed)
        path, prec = case["path"], case["prec"]
        if path in ("blocks", "blocks_local"):
            self.plans = [self.ctx.block_plan(case["op"], prec)]
        else:
            algo = path if path in ("tree", "direct") else "egraph"
            self.plans = [self.ctx.plan_operator(op, algo, prec) for op in case["op"].split(",")]
        self.C = [torch.zeros(sets, T, dtype=torch.complex128, device="cuda") for sets, T, _ in _geometries(case)
                  for _ in self.plans]
        sets, T, V3 = _geometries(case)[0]
        self.site_out = torch.zeros(sets, T, V3, dtype=torch.complex128, device="cuda") if case["sites"] else None
        if path == "host":
            self.fields = [tuple(f.cpu().pin_memory() for f in pair) for pair in self.fields]
            self.C = [torch.zeros(sets, T, dtype=torch.complex128).pin_memory()]
        if path == "batch":
            self.items = []
            for k, ((U, D), (sets, T, V3)) in enumerate(zip(self.fields, _geometries(case))):
                for q, plan in enumerate(self.plans):
                    self.items.append(dict(plan=plan.handle, U=U, D=D, n_sets=sets, T=T, V3=V3,
                                           C=self.C[k * len(self.plans) + q]))
            abi.mbc_batch_reserve(self.ctx.handle, self.items)

    def __del__(self):
        if getattr(self, "ctx", None) is not None:
            self.ctx.close()


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    case, plan = state.case, state.plans[0]
    U, D = state.fields[0]
    C, path, p = state.C[0], case["path"], _momentum(case)
    if path == "batch":
        state.ctx.batch(state.items)
        return list(state.C)
    if path == "host":
        plan.correlator_host(U, D, C)
    elif path == "blocks":
        plan.correlator(U, D, C, _extent(case["V3"]), p)
    elif path == "blocks_local":
        plan.correlator_local(U, D, C)
    elif p:
        plan.correlator_momentum(U, D, C, _extent(case["V3"]), p, state.site_out)
    else:
        plan.correlator(U, D, C, state.site_out)
    return [C] if state.site_out is None else [C, state.site_out]


def work(case):
    n_bytes = n_flops = 0.0
    for sets, T, V3 in _geometries(case):
        n = sets * T * V3
        n_bytes += n * 2 * 144 * 16
        for op in case["op"].split(","):
            n_bytes += sets * T * 16 + (n * 16 if case["sites"] else 0)
            if case["path"] in ("blocks", "blocks_local"):
                site, tree = BLOCK_FLOPS[op]
                n_flops += n * site + (sets * T if case["path"] == "blocks" else n) * tree
            else:
                algo = case["path"] if case["path"] in ("tree", "direct") else "egraph"
                n_flops += n * FLOPS[algo, op]
    return {"bytes": n_bytes, "flops": n_flops}


def tolerance(case):
    # FP32 with its guards (C(t) is guarded at 1e-6 of each slice; 3e-7 seen), double-float
    # (1e-13 seen) and double (5e-16 seen).  At nonzero momentum the nearly equal sites of a
    # noisy slice cancel to NOISE / sqrt(V3) of their size, and the rounding errors stay
    # (double-float: 1e-11 seen); FP32 recomputes those sites.
    rel = {"fp32": 2e-6, "mixed": 1e-12, "fp64": 1e-13}[case["prec"]]
    return {"rel": rel * 1e4 if case["noise"] and _momentum(case) and case["prec"] != "fp32" else rel}


# ------------------------------------------------------------------ the sums in 64 bits
def _matmul(a, b):
    return [[sum(a[i][k] * b[k][j] for k in range(4)) for j in range(4)] for i in range(4)]


def _gammas():
    """C gamma_5 and C gamma_5 (1 +- gamma_4) / 2 in the Dirac basis with C = gamma_4 gamma_2."""
    s = ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])
    g = []
    for k in range(3):
        m = [[0] * 4 for _ in range(4)]
        for i in range(2):
            for j in range(2):
                m[i][2 + j] = -1j * s[k][i][j]
                m[2 + i][j] = 1j * s[k][i][j]
        g.append(m)
    g4 = [[(1 if i < 2 else -1) if i == j else 0 for j in range(4)] for i in range(4)]
    g5 = _matmul(_matmul(g[0], g[1]), _matmul(g[2], g4))
    cg5 = _matmul(_matmul(g4, g[1]), g5)
    plus = [[(1 if i == j else 0) * (1 if i < 2 else 0) for j in range(4)] for i in range(4)]
    minus = [[(1 if i == j else 0) * (0 if i < 2 else 1) for j in range(4)] for i in range(4)]
    nz = lambda m: [(i, j, m[i][j]) for i in range(4) for j in range(4) if m[i][j] != 0]
    return {"": nz(cg5), "+": nz(_matmul(cg5, plus)), "-": nz(_matmul(cg5, minus))}


# sink operators: products (coefficient, baryons), the first two tied with C gamma_5 when
# there are two or more; a baryon is (flavour of its like quarks, projection)
_PRODUCTS = {
    "proton": (1.0, [(1, [("u", "")])]),
    "dinucleon_I": (1.0, [(1, [("d", ""), ("u", "")])]),
    "he3_I": (1.0, [(1, [("u", "-"), ("d", "+"), ("u", "+")])]),
    "he3_II_s": (2.0 / math.sqrt(6.0), [(1, [("u", "-"), ("d", "+"), ("u", "+")]), (-1, [("u", "+"), ("d", "+"), ("u", "-")]),
                                        (1, [("u", "+"), ("u", "-"), ("d", "+")])]),
}
_PERM3 = [((0, 1, 2), 1), ((1, 2, 0), 1), ((2, 0, 1), 1), ((0, 2, 1), -1), ((2, 1, 0), -1), ((1, 0, 2), -1)]


def _spins(n_baryons):
    """Per free index j: (spins of the baryons, weight)."""
    tie = _gammas()[""]
    if n_baryons == 1:
        return [[((j,), 1)] for j in range(2)]
    if n_baryons == 2:
        return [[((a, b), w) for a, b, w in tie]]
    return [[((a, b, j), w) for a, b, w in tie] for j in range(2)]


def _parity(seq):
    return -1 if sum(seq[i] > seq[k] for i in range(len(seq)) for k in range(i + 1, len(seq))) % 2 else 1


def _canonical(op):
    """Per free index: {(ascending up set, ascending down set): weight} of the sink operator,
    its normalisation left out (the free index runs over the two projected spins)."""
    gam = _gammas()
    out = [dict() for _ in range(1 if op == "dinucleon_I" else 2)]
    for coef, baryons in _PRODUCTS[op][1]:
        for j, ties in enumerate(_spins(len(baryons))):
            for spins, w in ties:
                parts = []
                for (q, proj), alpha in zip(baryons, spins):
                    other = "d" if q == "u" else "u"
                    parts.append([(sgn * g, ((q, 3 * be + c[0]), (other, 3 * ga + c[1]), (q, 3 * alpha + c[2])))
                                  for c, sgn in _PERM3 for be, ga, g in gam[proj]])
                for pick in itertools.product(*parts):
                    quarks = [f for _, fs in pick for f in fs]
                    keys = [(0 if f == "u" else 1, i) for f, i in quarks]
                    if len(set(keys)) < len(keys):
                        continue
                    weight = coef * w * _parity(keys)
                    for x, _ in pick:
                        weight = weight * x
                    k = (tuple(sorted(i for f, i in keys if f == 0)), tuple(sorted(i for f, i in keys if f == 1)))
                    out[j][k] = out[j].get(k, 0) + weight
    return [{k: w for k, w in d.items() if w != 0} for d in out]


def _minors(M, n, rows, cols):
    """det M[R, C] for every R in rows and C in cols: Laplace expansion along the last column."""
    dev = M.device
    T = torch.ones(M.shape[0], 1, 1, dtype=M.dtype, device=dev)
    prev = [()]
    for k in range(1, n + 1):
        sets = list(itertools.combinations(range(12), k))
        R, C = (rows, cols) if k == n else (sets, sets)
        at = {s: i for i, s in enumerate(prev)}
        last = torch.tensor([c[-1] for c in C], device=dev)
        below = torch.tensor([at[c[:-1]] for c in C], device=dev)
        new = None
        for i in range(k):
            r = torch.tensor([s[i] for s in R], device=dev)
            child = torch.tensor([at[s[:i] + s[i + 1:]] for s in R], device=dev)
            t = M[:, r][:, :, last] * T[:, child][:, :, below]
            t = t if (i + k - 1) % 2 == 0 else -t
            new = t if new is None else new.add_(t)
        T, prev = new, sets
    return T


def _site_values(op, U, D):
    """C_x of every site (U, D: [sites, 12, 12]) without the operator's normalisation."""
    dev = U.device
    sink = _canonical(op)
    rows = [sorted({k[f] for d in sink for k in d}) for f in range(2)]
    n = [len(rows[0][0]), len(rows[1][0])]
    out = []
    for u, d in zip(U.split(128), D.split(128)):
        A, B = _minors(u, n[0], rows[0], rows[0]), _minors(d, n[1], rows[1], rows[1])
        c = torch.zeros(u.shape[0], dtype=torch.complex128, device=dev)
        for terms in sink:
            ia = torch.tensor([rows[0].index(k[0]) for k in terms], device=dev)
            ib = torch.tensor([rows[1].index(k[1]) for k in terms], device=dev)
            w = torch.tensor([complex(x) for x in terms.values()], dtype=torch.complex128, device=dev)
            pairs = A[:, ia][:, :, ia].mul_(B[:, ib][:, :, ib])
            c += torch.matmul(torch.matmul(pairs, w.conj()), w)
        out.append(c)
    q = n[0] + n[1]
    return torch.cat(out) * (-1) ** (q * (q - 1) // 2)


def _phases(p, V3, dev):
    """e^{-i p.x 2 pi / L} of a slice's sites."""
    if p is None:
        return torch.ones(V3, dtype=torch.complex128, device=dev)
    L = _extent(V3)
    x = torch.arange(V3, device=dev)
    k = (p[0] * (x % L) + p[1] * ((x // L) % L) + p[2] * (x // (L * L))) % L
    a = -2.0 * math.pi / L * k.to(torch.float64)
    return torch.complex(torch.cos(a), torch.sin(a))


def _projected_blocks(Q1, Q2, proj, phase):
    """F[s1, s2, s3, alpha] of one baryon type, summed over the sites with the phase."""
    u, d = Q1.view(-1, 4, 3, 12), Q2.view(-1, 4, 3, 12)        # [x, spin, colour, source]
    F = torch.zeros(12, 12, 12, 4, dtype=torch.complex128, device=Q1.device)
    for (a, b, c), sgn in _PERM3:
        diq = sum(g * torch.einsum("xs,xt->xst", u[:, be, a], d[:, ga, b]) for be, ga, g in _gammas()[proj])
        t = torch.matmul((diq * (sgn * phase).view(-1, 1, 1)).reshape(-1, 144).t(), u[:, :, c].reshape(-1, 48))
        t = t.view(12, 12, 4, 12)                              # [s, s2, alpha, s1]
        F += t.permute(3, 1, 0, 2) - t.permute(0, 1, 3, 2)
    return F


def _assignments(baryons, n_u, n_d):
    """Every way to hand the source slots to the sink baryons in the order (q1, q2, q1): [(slots, sign)]."""
    out = []

    def rec(i, fu, fd, slots):
        if i == len(baryons):
            order = [s for b in slots for s in b]
            out.append((slots, _parity(order) * (-1) ** (len(baryons) * (len(baryons) - 1) // 2)))
            return
        like, other = (fu, fd) if baryons[i][0] == "u" else (fd, fu)
        for a, c in itertools.combinations(like, 2):
            for b in other:
                l2, o2 = tuple(x for x in like if x not in (a, c)), tuple(x for x in other if x != b)
                rec(i + 1, *((l2, o2) if baryons[i][0] == "u" else (o2, l2)), slots + [(a, b, c)])

    rec(0, tuple(range(n_u)), tuple(range(n_u, n_u + n_d)), [])
    return out


def _projected_values(op, U, D, phase):
    """The block form of one slice: sum over assignments of products of projected blocks."""
    dev = U.device
    types = sorted({b for _, bs in _PRODUCTS[op][1] for b in bs})
    F = {t: _projected_blocks(*((U, D) if t[0] == "u" else (D, U)), t[1], phase) for t in types}
    total = torch.zeros((), dtype=torch.complex128, device=dev)
    source = _canonical(op)
    for coef, baryons in _PRODUCTS[op][1]:
        asg = _assignments(baryons, len(next(iter(source[0]))[0]), len(next(iter(source[0]))[1]))
        sign = torch.tensor([s for _, s in asg], dtype=torch.complex128, device=dev)
        for j, ties in enumerate(_spins(len(baryons))):
            src = torch.tensor([k[0] + k[1] for k in source[j]], device=dev)
            w = torch.tensor([complex(x) for x in source[j].values()], dtype=torch.complex128, device=dev).conj()
            for spins, tw in ties:
                prod = None
                for i, (b, alpha) in enumerate(zip(baryons, spins)):
                    s = torch.tensor([x[i] for x, _ in asg], device=dev)
                    f = F[b][src[:, s[:, 0]], src[:, s[:, 1]], src[:, s[:, 2]], alpha]
                    prod = f if prod is None else prod * f
                total += coef * complex(tw) * (w @ (prod @ sign))
    return total


def exact(case, seed):
    out = []
    for (U, D), (sets, T, V3) in zip(_fields(case, seed), _geometries(case)):
        phase = _phases(_momentum(case), V3, U.device)
        for op in case["op"].split(","):
            if op not in _PRODUCTS:           # the printed operators that vanish identically
                out.append(torch.zeros(sets, T, dtype=torch.complex128))
                continue
            norm = _PRODUCTS[op][0] ** 2
            if case["path"] == "blocks":
                C = [_projected_values(op, U[s, t], D[s, t], phase) for s in range(sets) for t in range(T)]
                out.append((norm * torch.stack(C)).view(sets, T).cpu())
                continue
            c = norm * _site_values(op, U.view(-1, 12, 12), D.view(-1, 12, 12)).view(sets, T, V3)
            out.append((c * phase).sum(dim=2).cpu())
            if case["sites"]:
                out.append(c.cpu())
    return out
