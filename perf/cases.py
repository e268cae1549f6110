"""Performance cases of the contraction library.

A case is one ``contract`` call as a program makes it for a set of gauge
configurations: the propagator field is on the GPU, the term lists were built
once, and every pass evaluates the correlators of the call's nuclei. The
workloads are those of ``bench.py`` (nuclei, lattices, storage, momenta), cut
in the number of sites where a full lattice would take minutes, plus ragged
lattices, several configurations, momenta and time-slice sub-ranges.

Propagators: Gaussian draws (``eps`` = 0) where the FP64 correlator keeps its
digits on them, near-identity draws 1 + eps R otherwise (propagators dominated
by their diagonal); both decay as exp(-lam t).

The mixed path carries FP32 accuracy; a program that asks for it keeps the
correlators as complex64, so its passes end with that conversion. FP64 passes
return the library's complex128.
"""
import functools
import itertools
import math

import numpy as np
import torch

import paper_1301_4895_gb300 as mbc

DEV = "cuda:0"
MOMENTA = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 1, 1)]
PAIRS = ((0, 1), (0, 2), (1, 2), (0, 3), (1, 3), (2, 3))  # ascending pairs of 4 spins, as the library orders them
HE4_SPINS = (0, 1, 0, 1)
BE8_SPINS = (0, 1, 2, 3, 0, 1, 2, 3)


def _all_components(n_p, n_n, dim):
    """Every (sink, source) pair of independent spin sets, as the library orders them."""
    def sets(n):
        return sorted(itertools.combinations(range(dim), n), key=lambda s: sum(1 << i for i in s))
    spins = [p + n for p in sets(n_p) for n in sets(n_n)]
    return [(a, b) for a in spins for b in spins]


def _nucleus(n_p, n_n, dim, comps=None, n_src=1, n_snk=1):
    return {"n_p": n_p, "n_n": n_n, "dim": dim, "n_src": n_src, "n_snk": n_snk, "listed": comps is not None,
            "comps": comps if comps is not None else _all_components(n_p, n_n, dim)}


PN, HE3, HE4 = _nucleus(1, 1, 2), _nucleus(2, 1, 2), _nucleus(2, 2, 2)
HE4_REL = _nucleus(2, 2, 4, [(HE4_SPINS, HE4_SPINS)])
HE4_ALL = _nucleus(2, 2, 4)
BE8 = _nucleus(4, 4, 4, [(BE8_SPINS, BE8_SPINS)])
HE4_TWO = _nucleus(2, 2, 2, [(p + q, (0, 2, 0, 2)) for p in PAIRS for q in PAIRS], n_src=2, n_snk=2)

# the term lists of a call; "joined": one list, several nuclei on one path
CALLS = {
    "pn": [PN],
    "he3he4": [HE3, HE4],
    "joined": [HE3, HE4],
    "batched": [PN, HE3, HE4, HE4_REL],
    "he4rel": [HE4_REL],
    "he4all": [HE4_ALL],
    "be8": [BE8],
    "he4rel_blocks": [HE4_REL],
    "he4two_blocks": [HE4_TWO],
}


def _case(name, call, prec, store, dims, nt, cfgs=1, moms=1, t0=0, eps=0.0, lam=0.4):
    lz, ly, lx = dims
    c = {"name": name, "call": call, "prec": prec, "store": store, "cfgs": cfgs, "nt": nt, "lz": lz, "ly": ly, "lx": lx,
         "moms": moms, "t0": t0, "eps": eps, "lam": lam}
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # the smallest call in use: all deuteron components on a test lattice, where latency counts
        _case("pn_small", "pn", "fp64", "c128", (4, 4, 4), 8, lam=0.5),
        # the benchmark's default workload: light nuclei with nonrelativistic operators, a whole configuration
        _case("he3he4", "he3he4", "fp64", "c128", (16, 16, 16), 32),
        _case("he3he4_mixed", "he3he4", "mixed", "c128", (16, 16, 16), 32, eps=0.05),
        # the same nuclei on one recursion path: ragged lattice, FP32 storage, several configurations and momenta
        _case("joined_ragged", "joined", "fp64", "c64", (9, 11, 13), 5, cfgs=2, moms=3, t0=1, eps=0.05),
        # nuclei of both operator kinds in one call over configurations and time slices
        _case("batched", "batched", "fp64", "c64", (8, 8, 8), 2, cfgs=2, eps=0.05),
        # relativistic 4He, one spin component, the case most relativistic runs need
        _case("he4rel_mixed", "he4rel", "mixed", "c128", (16, 16, 16), 4, eps=0.05),
        # relativistic 4He, every spin component
        _case("he4all", "he4all", "fp64", "c128", (4, 4, 4), 1, eps=0.05),
        _case("he4all_mixed", "he4all", "mixed", "c128", (8, 8, 8), 1, eps=0.05),
        # 8Be, the largest nucleus, stored in FP32
        _case("be8", "be8", "fp64", "c64", (4, 4, 4), 1, eps=0.02),
        _case("be8_mixed", "be8", "mixed", "c64", (8, 8, 8), 1, eps=0.02),
        # every baryon projected to a momentum before the recursion (the source method's own use)
        _case("he4rel_blocks", "he4rel_blocks", "fp64", "c128", (16, 16, 16), 4, moms=4, eps=0.05),
        # two quark sources and two sink functions with projected blocks
        _case("he4two_blocks_mixed", "he4two_blocks", "mixed", "c128", (16, 16, 16), 16, moms=2, eps=0.05),
    ]


# sites (configurations x evaluated slices x lattice) that a drawn case spans, per arithmetic
RANGES = {
    "pn": {"fp64": (256, 131072), "mixed": (256, 131072)},
    "he3he4": {"fp64": (256, 131072), "mixed": (256, 131072)},
    "joined": {"fp64": (256, 131072), "mixed": (256, 131072)},
    "batched": {"fp64": (64, 2048), "mixed": (256, 16384)},
    "he4rel": {"fp64": (64, 2048), "mixed": (256, 16384)},
    "he4all": {"fp64": (8, 64), "mixed": (32, 512)},
    "be8": {"fp64": (8, 64), "mixed": (32, 512)},
    "he4rel_blocks": {"fp64": (256, 16384), "mixed": (1024, 65536)},
    "he4two_blocks": {"fp64": (256, 16384), "mixed": (1024, 65536)},
}


def draw(rng):
    call = rng.choice(sorted(RANGES))
    prec = rng.choice(["fp64", "mixed"])
    lo, hi = RANGES[call][prec]
    while True:
        sites = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        # extents around the cube root of the share of one slice, odd and unequal ones among them
        slabs = max(1, min(int(math.exp(rng.uniform(0.0, math.log(24)))), int(sites / 8)))
        if call in ("he4all", "be8"):
            slabs = 1
        edge = (sites / slabs) ** (1.0 / 3.0)
        dims = tuple(max(1, min(24, int(round(edge * rng.uniform(0.7, 1.4))))) for _ in range(3))
        cfgs = 2 if slabs >= 2 and rng.random() < 0.3 else 1
        nt = max(1, slabs // cfgs)
        if lo // 2 <= cfgs * nt * dims[0] * dims[1] * dims[2] <= hi:
            break
    t0 = 1 if rng.random() < 0.25 else 0
    moms = rng.choice([2, 4]) if call == "he4two_blocks" else rng.choice([1, 1, 2, 3, 4])
    near = call in ("be8", "he4all", "he4rel", "batched", "he4rel_blocks", "he4two_blocks") or prec == "mixed"
    eps = 0.02 if call == "be8" else 0.05 if near or rng.random() < 0.5 else 0.0
    return _case(None, call, prec, rng.choice(["c128", "c64"]), dims, nt + t0, cfgs=cfgs, moms=moms, t0=t0, eps=eps)


# ---- what a program has in hand ------------------------------------------------


@functools.lru_cache(maxsize=None)
def _lists(call):
    """The term lists of a call, built once per process (as a program keeps them)."""
    nuclei = CALLS[call]
    if call == "joined":
        return (mbc.build_combined([{"n_p": n["n_p"], "n_n": n["n_n"]} for n in nuclei], nuclei[0]["dim"], path=[0, 0, 1, 1]),)
    return tuple(mbc.build_term_list(n["n_p"], n["n_n"], n["dim"], spins=n["comps"] if n["listed"] else None,
                                     n_sources=n["n_src"], n_sinks=n["n_snk"]) for n in nuclei)


def _field(case, seed):
    """(cfgs, nt, Lz, Ly, Lx, [sources,] 12, 12), drawn on the GPU."""
    n_src = CALLS[case["call"]][0]["n_src"]
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    shape = (case["cfgs"], case["nt"], case["lz"], case["ly"], case["lx"]) + ((n_src,) if n_src > 1 else ()) + (12, 12)
    s = torch.view_as_complex(torch.randn(shape + (2,), dtype=torch.float64, device=DEV, generator=g))
    if case["eps"]:
        s.mul_(case["eps"]).add_(torch.eye(12, dtype=torch.complex128, device=DEV))
    t = torch.arange(case["nt"], device=DEV, dtype=torch.float64)
    s.mul_(torch.exp(-case["lam"] * t).reshape((1, -1) + (1,) * (len(shape) - 2)))
    return s if case["store"] == "c128" else s.to(torch.complex64)


def prepare(case, seed):
    return {"field": _field(case, seed), "lists": _lists(case["call"]), "moms": MOMENTA[:case["moms"]], "t0": case["t0"],
            "prec": mbc.MIXED if case["prec"] == "mixed" else mbc.FP64,
            "sink": mbc.SINK_BLOCK_MOMENTUM if case["call"].endswith("blocks") else mbc.SINK_POINT}


def run(state):
    # on torch's current stream, where the field was made and the result is used
    out = mbc.contract(state["field"], state["lists"], precision=state["prec"], moms=state["moms"], t0=state["t0"],
                       sink=state["sink"], stream=torch.cuda.current_stream())
    return out.to(torch.complex64) if state["prec"] == mbc.MIXED else out


def _out_shape(case):
    nuclei = CALLS[case["call"]]
    n_snk = nuclei[0]["n_snk"]
    counts = [sum(len(n["comps"]) for n in nuclei)] if case["call"] == "joined" else [len(n["comps"]) for n in nuclei]
    return (case["cfgs"], len(counts), case["nt"] - case["t0"], case["moms"] // n_snk, max(counts))


def work(case):
    """Bytes: the entries of every propagator that the operators reach, and the
    output. Floating-point operations: no form of the correlator takes less
    than one elimination of a site's tile and one multiply-add per nonzero
    entry of the source tensors L (per item for projected blocks, whose sites
    take one multiply-add per block entry and momentum instead)."""
    nuclei = CALLS[case["call"]]
    sites = case["cfgs"] * (case["nt"] - case["t0"]) * case["lz"] * case["ly"] * case["lx"]
    rows = 3 * max(n["dim"] for n in nuclei)
    cols = rows * nuclei[0]["n_src"]
    n_l = sum(tl.stats()["n_l_total"] for tl in _lists(case["call"]))
    out = math.prod(_out_shape(case))
    if case["call"].endswith("blocks"):
        block = (rows // 3) * (cols * (cols - 1) // 2) * cols
        items = case["cfgs"] * (case["nt"] - case["t0"]) * case["moms"] // nuclei[0]["n_snk"]
        flops = 8.0 * block * case["moms"] * sites + 8.0 * n_l * items
    else:
        flops = sites * (8.0 * rows ** 3 / 3 + 8.0 * n_l)
    return {"bytes": float(sites * rows * cols * (16 if case["store"] == "c128" else 8) + 16 * out), "flops": flops}


# ---- the same correlators from their definition, in FP64 -------------------------
# Quark sets are bit masks. A nucleus is the antisymmetric product of its
# baryons' blocks; C = sum over quark sets of F(sink) L(source), where the
# source tensor L is F of a unit propagator.


@functools.lru_cache(maxsize=None)
def _subsets(n, k):
    return [sum(1 << i for i in c) for c in itertools.combinations(range(n), k)]


@functools.lru_cache(maxsize=None)
def _place(n, k):
    return {m: i for i, m in enumerate(_subsets(n, k))}


@functools.lru_cache(maxsize=None)
def _sign(x, y):
    """(-1)^(pairs i in x, j in y with i > j)"""
    return -1 if sum(bin(x >> (j + 1)).count("1") for j in range(y.bit_length()) if y >> j & 1) % 2 else 1


@functools.lru_cache(maxsize=None)
def _splits(n, whole, k):
    """Places of the k-subsets of a mask, of their complements in it, and the signs."""
    bits = [i for i in range(n) if whole >> i & 1]
    sub = [sum(1 << i for i in c) for c in itertools.combinations(bits, k)]
    return (np.array([_place(n, k)[s] for s in sub]), np.array([_place(n, len(bits) - k)[whole ^ s] for s in sub]),
            np.array([_sign(s, whole ^ s) for s in sub], dtype=np.float64))


def _blocks(tile, dim):
    """f[alpha, pair * column, site] of tiles (site, 3 dim rows, columns): sum over colour
    eps eps' S S S with Gamma_1 = 1, Gamma_2 = C gamma_5, antisymmetric in the pair."""
    s = tile.reshape(tile.shape[0], dim, 3, -1)
    n = s.shape[-1]
    q = torch.zeros((tile.shape[0], 3, n, n), dtype=tile.dtype, device=tile.device)
    for s2, s3, v in ((0, 1, -1), (1, 0, 1), (2, 3, -1), (3, 2, 1))[:dim]:
        for c in range(3):
            for c2, c3, e in (((c + 1) % 3, (c + 2) % 3, 1), ((c + 2) % 3, (c + 1) % 3, -1)):
                q[:, c] += v * e * s[:, s2, c2, :, None] * s[:, s3, c3, None, :]
    f = torch.einsum("xaci,xcjk->aijkx", s, q)
    pairs = list(itertools.combinations(range(n), 2))
    i, j = (torch.tensor(v, device=tile.device) for v in zip(*pairs))
    return (f[:, i, j] - f[:, j, i]).reshape(dim, len(pairs) * n, -1)


def _product(f, spins, n):
    """Ordered product of one or two blocks: values [u set * d set, site] of proton type."""
    if len(spins) == 1:
        return f[spins[0]]
    a = [_splits(n, m, 2) for m in _subsets(n, 4)]
    e = np.array([[i for i in range(n) if m >> i & 1] for m in _subsets(n, 2)])
    p = torch.from_numpy(np.stack([x[0] for x in a])).to(f.device)
    r = torch.from_numpy(np.stack([x[1] for x in a])).to(f.device)
    sg = torch.from_numpy(np.stack([x[2] for x in a])).to(f.device)
    e1, e2 = torch.from_numpy(e[:, 0]).to(f.device), torch.from_numpy(e[:, 1]).to(f.device)
    x, y = f[spins[0]].reshape(-1, n, f.shape[-1]), f[spins[1]].reshape(-1, n, f.shape[-1])
    out = 0
    for j in range(6):
        xs, ys = x[p[:, j]], y[r[:, j]]
        out = out + sg[:, j, None, None] * (xs[:, e1] * ys[:, e2] - xs[:, e2] * ys[:, e1])
    return out.reshape(-1, f.shape[-1])


@functools.lru_cache(maxsize=None)
def _source(call, which):
    """Keys z of a nucleus' source tensors and L[source spins, z], from unit propagators."""
    nu = CALLS[call][which]
    n_p, n_n, dim, n_src = nu["n_p"], nu["n_n"], nu["dim"], nu["n_src"]
    n = 3 * dim * n_src
    f = []
    for chi in range(dim * n_src):  # baryon index spin * sources + source: all quarks from that source
        unit = torch.zeros((1, 3 * dim, n), dtype=torch.complex128)
        for r in range(3 * dim):
            unit[0, r, n_src * r + chi % n_src] = 1
        f.append(_blocks(unit, dim)[chi // n_src])
    f = torch.stack(f)
    spins = sorted({b for _, b in nu["comps"]})
    rows = []
    for b in spins:
        part = []
        for sel, k in ((b[:n_p], n_p), (b[n_p:], n_n)):
            v = _product(f, sel, n)[:, 0].real.numpy()
            nd = len(_subsets(n, k))
            part.append([(_subsets(n, 2 * k)[i // nd], _subsets(n, k)[i % nd], v[i]) for i in np.nonzero(v)[0]])
        row = {}
        for a, e, v in part[0]:
            for d, u, w in part[1]:  # neutron type: the pairs are d quarks
                if not a & u and not e & d:
                    key = (a | u, e | d)
                    row[key] = row.get(key, 0.0) + v * w * _sign(a, u) * _sign(e, d)
        rows.append(row)
    keys = sorted({k for r in rows for k, v in r.items() if v})
    at = {k: i for i, k in enumerate(keys)}
    L = np.zeros((len(spins), len(keys)))
    for i, r in enumerate(rows):
        for k, v in r.items():
            if v:
                L[i, at[k]] = v
    ip, iq, sg = [], [], []
    for U, D in keys:
        a, u, su = _splits(n, U, 2 * n_p)
        e, d, sd = _splits(n, D, n_p)
        ip.append((a[:, None] * len(_subsets(n, n_p)) + e[None, :]).reshape(-1))
        iq.append((d[None, :] * len(_subsets(n, n_n)) + u[:, None]).reshape(-1))
        sg.append((su[:, None] * sd[None, :]).reshape(-1))
    to = [torch.from_numpy(np.stack(v)).to(DEV) for v in (ip, iq, sg)]
    return spins, torch.from_numpy(L).to(DEV).to(torch.complex128), to


def _components(call, which, f):
    """C[component, site or item] of one nucleus from blocks f[index, entries, site]."""
    nu = CALLS[call][which]
    n = 3 * nu["dim"] * nu["n_src"]
    n_p = nu["n_p"]
    spins, L, (ip, iq, sg) = _source(call, which)
    C = torch.empty((len(nu["comps"]), f.shape[-1]), dtype=torch.complex128, device=DEV)
    parts = {}
    for a, _ in nu["comps"]:
        for s in (a[:n_p], a[n_p:]):
            if s not in parts:
                parts[s] = _product(f, s, n)
    step = max(1, (1 << 25) // (ip.shape[1] * f.shape[-1]))
    for snk in sorted({a for a, _ in nu["comps"]}):
        P, N = parts[snk[:n_p]], parts[snk[n_p:]]
        acc = 0
        for z in range(0, ip.shape[0], step):
            F = (P[ip[z:z + step]] * N[iq[z:z + step]] * sg[z:z + step, :, None]).sum(1)
            acc = acc + L[:, z:z + step] @ F
        for i, (a, b) in enumerate(nu["comps"]):
            if a == snk:
                C[i] = acc[spins.index(b)]
    return C


def _tile(x, dim, n_src):
    """(site, 3 dim, 3 dim sources) tiles of (site, [source,] 12, 12) propagators."""
    r = 3 * dim
    if n_src == 1:
        return x[..., :r, :r].reshape(-1, r, r)
    x = x[..., :r, :r].reshape(-1, n_src, r, r)
    return x.permute(0, 2, 3, 1).reshape(-1, r, r * n_src)


def exact(case, seed):
    nuclei, call = CALLS[case["call"]], case["call"]
    shape = _out_shape(case)
    cfgs, _, n_t, n_out, _ = shape
    field = _field(case, seed).to(torch.complex128)[:, case["t0"]:]
    v3 = case["lz"] * case["ly"] * case["lx"]
    lat = [torch.arange(case[k], device=DEV, dtype=torch.float64) / case[k] for k in ("lz", "ly", "lx")]
    turns = torch.stack([(m[2] * lat[0][:, None, None] + m[1] * lat[1][None, :, None] + m[0] * lat[2][None, None, :]).reshape(-1)
                         for m in MOMENTA[:case["moms"]]])
    phase = torch.polar(torch.ones_like(turns), -2 * math.pi * turns)  # [mom, site]
    out = torch.zeros(shape, dtype=torch.complex128, device=DEV)
    step = {2: 4096, 4: 64}[max(n["dim"] for n in nuclei)]
    if call == "he4two_blocks":
        step = 512
    for cfg in range(cfgs):
        if call.endswith("blocks"):
            nu = nuclei[0]
            n_snk, f_items = nu["n_snk"], []
            for t in range(n_t):
                flat = field[cfg, t].reshape((v3,) + tuple(field.shape[5:]))
                f = 0
                for x in range(0, v3, step):
                    b = _blocks(_tile(flat[x:x + step], nu["dim"], nu["n_src"]), nu["dim"])
                    f = f + torch.einsum("aex,qx->qae", b, phase[:, x:x + step])
                # sink index spin * functions + function, one momentum per function
                f = f.reshape((n_out, n_snk) + tuple(f.shape[1:])).permute(0, 2, 1, 3)
                f_items.append(f.reshape(n_out, -1, f.shape[-1]))
            items = torch.cat(f_items).permute(1, 2, 0).contiguous()  # [index, entries, t * group]
            C = torch.cat([_components(call, 0, items[..., i:i + 32].contiguous()) for i in range(0, items.shape[-1], 32)], 1)
            out[cfg, 0, :, :, :C.shape[0]] = C.reshape(C.shape[0], n_t, n_out).permute(1, 2, 0)
            continue
        for t in range(n_t):
            flat = field[cfg, t].reshape(v3, 12, 12)
            for x in range(0, v3, step):
                ph = phase[:, x:x + step]
                if call == "be8":  # every source state taken: C = L^2 det S_u det S_d
                    C = 1814400.0 ** 2 * torch.linalg.det(flat[x:x + step])[None] ** 2
                    out[cfg, 0, t] += ph @ C.T
                    continue
                f = {d: _blocks(_tile(flat[x:x + step], d, 1), d) for d in {n["dim"] for n in nuclei}}
                at = 0
                for i, nu in enumerate(nuclei):
                    C = _components(call, i, f[nu["dim"]])
                    li, c0 = (0, at) if call == "joined" else (i, 0)
                    out[cfg, li, t, :, c0:c0 + C.shape[0]] += ph @ C.T
                    at += C.shape[0]
    return out
