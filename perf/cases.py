"""Workloads of the RI-MP2 engine as a user's program runs them, through the package's
public calls (`rimp2.Engine`, `rimp2.MBEAssembly`, the screen's training and prediction
calls, `rimp2.zvector`), with seeded inputs, the work of one pass and 64-bit results of the
same inputs from plain torch.

Sizes are those of the package's own workloads: the tiny (10, 40, 150) and the large
(100, 500, 1500) single fragment, monomers / dimers / trimers of the 64-monomer 40-bohr MBE3
system (nocc 8..20 a monomer, nvir = 4 nocc, naux = 3 (nocc + nvir)), the learned screen's
512-sample training steps and 20,000-trimer predictions, the gradient step after the
densities.  Single fragments also take ragged sizes (ratios of a real basis set are not
multiples of anything).
"""
from __future__ import annotations

import itertools
import math

import torch

from paper_2410_21888_gb300 import rimp2

SIGMA = 0.05      # spread of B
DECAY = 3.0       # bohr; inter-monomer blocks of B fall off as exp(-distance / DECAY)
DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------------------ the cases

def listed():
    return [
        # one small molecule, plain FP64: launch latency and half-empty tiles count
        {"name": "fragment_small_fp64", "kind": "fragment", "precision": "fp64",
         "nocc": 10, "nvir": 40, "naux": 150},
        # the same molecule on the tensor-core path
        {"name": "fragment_small_bf16", "kind": "fragment", "precision": "bf16",
         "nocc": 10, "nvir": 40, "naux": 150},
        # one dimer-sized molecule in FP64 at a ragged size: the reference calculation that
        # audits of the faster paths recompute
        {"name": "fragment_mid_fp64", "kind": "fragment", "precision": "fp64",
         "nocc": 29, "nvir": 117, "naux": 437},
        # the largest single fragment the engine is quoted on
        {"name": "fragment_large_bf16", "kind": "fragment", "precision": "bf16",
         "nocc": 100, "nvir": 500, "naux": 1500},
        # a trimer-sized molecule on the FP8 path
        {"name": "fragment_mid_fp8", "kind": "fragment", "precision": "fp8",
         "nocc": 42, "nvir": 168, "naux": 630},
        # MBE3 level 1: every monomer of the system in one grouped FP64 plan
        {"name": "monomers_fp64", "kind": "batch", "precision": "fp64", "level": 1, "nfrag": 64,
         "grad": True},
        # MBE3 level 2: uneven dimers, energies and gradient intermediates, split path
        {"name": "dimers_bf16", "kind": "batch", "precision": "bf16", "level": 2, "nfrag": 40,
         "grad": True},
        # labels of the learned screen: trimer energies only, eight slices for V
        {"name": "trimer_energies_bf16", "kind": "batch", "precision": "bf16", "level": 3,
         "nfrag": 16, "grad": False},
        # MBE3 assembly: coefficient-weighted gather of all fragments' Gamma, P_ij, P_ab
        {"name": "assembly", "kind": "assembly", "monomers": 64, "box": 40.0, "r_dimer": 12.0,
         "r_trimer": 10.0},
        # one minibatch step of the screen's training: gradient and Adam update
        {"name": "screen_train_step", "kind": "train", "rows": 4500, "batch": 512},
        # screening a candidate list: features and predictions
        {"name": "screen_predict", "kind": "predict", "monomers": 256, "trimers": 22018},
        # the gradient step after the densities of a dimer-sized fragment (Gamma^P, L', L'',
        # Z-vector)
        {"name": "gradient_step", "kind": "gradient", "nocc": 30, "nvir": 120, "naux": 450},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["fragment", "fragment", "fragment", "batch", "batch", "assembly", "train",
                       "predict", "gradient"])
    if kind == "fragment":
        prec = rng.choice(["fp64", "bf16", "bf16", "fp8"])
        top = {"fp64": 36, "bf16": 92, "fp8": 60}[prec]
        o = _log_int(rng, 5, top)
        v = int(o * rng.uniform(3.0, 5.0)) + rng.randrange(0, 3)
        x = int((o + v) * rng.uniform(2.0, 3.0)) + rng.randrange(0, 3)
        return {"kind": kind, "precision": prec, "nocc": o, "nvir": v, "naux": x}
    if kind == "batch":
        level = rng.choice([1, 2, 3])
        prec = rng.choice(["bf16", "fp8"] + (["fp64"] if level == 1 else []))
        top = {1: 64, 2: 40, 3: 16}[level]
        return {"kind": kind, "precision": prec, "level": level, "nfrag": _log_int(rng, 2, top),
                "grad": prec == "fp64" or rng.random() < 0.6}
    if kind == "assembly":
        n = _log_int(rng, 6, 64)
        rd = rng.uniform(8.0, 12.0)
        return {"kind": kind, "monomers": n, "box": 10.0 * n ** (1.0 / 3.0), "r_dimer": rd,
                "r_trimer": rd * rng.uniform(0.6, 0.9)}
    if kind == "train":
        rows = _log_int(rng, 500, 20000)
        return {"kind": kind, "rows": rows, "batch": min(rows, _log_int(rng, 32, 2048))}
    if kind == "predict":
        return {"kind": kind, "monomers": _log_int(rng, 32, 256), "trimers": _log_int(rng, 500, 200000)}
    o = _log_int(rng, 4, 44)
    v = int(o * rng.uniform(3.0, 5.0)) + rng.randrange(0, 3)
    return {"kind": kind, "nocc": o, "nvir": v, "naux": int((o + v) * rng.uniform(2.0, 3.0)) + 1}


# ------------------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, n, lo, hi):
    return torch.rand(n, dtype=F64, device=DEV, generator=g) * (hi - lo) + lo


class _Frag:
    """One fragment's inputs, as `Engine.set_inputs` takes them."""

    def __init__(self, g, dims, parts=None, scale=None):
        o, v, x = dims
        self.eo = _uniform(g, o, -1.5, -0.3)
        self.ev = _uniform(g, v, 0.2, 3.0)
        self.B = torch.empty((o, v, x), dtype=F64, device=DEV)
        self.B.normal_(0.0, SIGMA, generator=g)
        if parts is not None:          # blocks of several monomers fall off with their distances
            ro, rv, rx = ([0] + list(itertools.accumulate(p[k] for p in parts)) for k in range(3))
            m = range(len(parts))
            for p, q, r in itertools.product(m, m, m):
                s = scale(sorted({p, q, r}))
                if s != 1.0:
                    self.B[ro[p]:ro[p + 1], rv[q]:rv[q + 1], rx[r]:rx[r + 1]] *= s


def _monomers(n, sizes):
    """n monomers' (nocc, nvir, naux); their sizes come from the case, not from the seed, so
    that every state of a case has the same shapes."""
    out = []
    for k in range(n):
        o = 8 + (((k + 1) * 2654435761 + sizes * 40503) >> 9) % 13
        out.append((o, 4 * o, 15 * o))
    return out


def _batch_parts(case):
    mono = _monomers(case["level"] * case["nfrag"], case["nfrag"])
    return [mono[case["level"] * f:case["level"] * (f + 1)] for f in range(case["nfrag"])]


def _dims(case):
    if case["kind"] == "fragment":
        return [(case["nocc"], case["nvir"], case["naux"])]
    return [tuple(sum(p[k] for p in parts) for k in range(3)) for parts in _batch_parts(case)]


def _fragments(case, seed):
    """The inputs of the case's fragments, one at a time."""
    g = _gen(seed)
    if case["kind"] == "fragment":
        yield _Frag(g, _dims(case)[0])
        return
    dist = torch.rand((case["nfrag"], 3), generator=torch.Generator().manual_seed(int(seed))) * 6 + 4
    for f, (dims, parts) in enumerate(zip(_dims(case), _batch_parts(case))):
        d = [float(t) for t in dist[f]]      # bohr, of the pairs (0,1), (0,2), (1,2)

        def scale(owners, d=d):
            return math.exp(-sum(d[a + b - 1] for a, b in itertools.combinations(owners, 2)) / DECAY)

        yield _Frag(g, dims, parts, scale)


def _geometry(n, box):
    """Monomer centroids in a box (fixed for a case: a system's geometry)."""
    return torch.rand((n, 3), dtype=F64, generator=torch.Generator().manual_seed(n)) * box


def _polymers(case):
    """Monomer sizes, fragments (monomers, dimers, trimers) and their MBE3 coefficients."""
    n = case["monomers"]
    d = torch.cdist(_geometry(n, case["box"]), _geometry(n, case["box"])).tolist()
    near = [[d[a][b] <= case["r_trimer"] for b in range(n)] for a in range(n)]
    pairs = [(a, b) for a in range(n) for b in range(a + 1, n) if d[a][b] <= case["r_dimer"]]
    trios = [(a, b, c) for a, b in pairs if near[a][b] for c in range(b + 1, n) if near[a][c] and near[b][c]]
    coeff = {(a,): 1 for a in range(n)}
    for p in pairs:
        coeff[p] = 1
        for a in p:
            coeff[(a,)] -= 1
    for t in trios:
        coeff[t] = 1
        for p in itertools.combinations(t, 2):
            coeff[p] -= 1
        for a in t:
            coeff[(a,)] += 1
    return _monomers(n, n), list(coeff), list(coeff.values())


def _pools(case, seed):
    """The fragments' Gamma, P_ij, P_ab in batch pools, and their offsets."""
    mono, frags, coeff = _polymers(case)
    off, at = [], [0, 0, 0]
    for f in frags:
        o, v, x = (sum(mono[m][k] for m in f) for k in range(3))
        off.append((tuple(at), (o, v, x)))
        at = [at[0] + o * v * x, at[1] + o * o, at[2] + v * v]
    g = _gen(seed)
    pools = [torch.empty(max(n, 1), dtype=F64, device=DEV).normal_(0.0, 1e-3, generator=g) for n in at]
    return mono, frags, coeff, off, pools


def _screen(case, seed):
    """Features, labels and a network in the middle of its training."""
    g = _gen(seed)
    n = case["rows"]
    base = torch.tensor([8, 10, 12, 8, 9, 10, -8, -7, -6], dtype=torch.float32, device=DEV)
    wide = torch.tensor([2, 2, 2, 3, 3, 3, 1.5, 1.5, 1.5], dtype=torch.float32, device=DEV)
    feats = base + wide * torch.randn((n, 9), device=DEV, generator=g)
    y = -3 - 0.4 * feats[:, 0] + 0.2 * feats[:, 6] + 0.05 * torch.randn(n, device=DEV, generator=g)
    P = rimp2.MLP_PARAMS
    m = torch.randn(P, device=DEV, generator=g) * 1e-3
    v = m * m + 1e-6 * torch.rand(P, device=DEV, generator=g)
    idx = torch.randperm(n, device=DEV, generator=g)[:case["batch"]].to(torch.int32)
    return {"feats": feats, "y": y, "idx": idx, "master": _network(g), "m": m, "v": v, "t": 100,
            "mean": feats.mean(0), "std": feats.std(0) + 1e-3}


_LAYERS = ((64, 9), (64, 64), (64, 64), (1, 64))


def _network(g):
    parts = []
    for o, i in _LAYERS:
        parts.append(torch.randn(o * i, device=DEV, generator=g) * math.sqrt(2.0 / i))
        parts.append(torch.randn(o, device=DEV, generator=g) * 0.05)
    return torch.cat(parts)


def _candidates(case, seed):
    """A monomer system, its candidate trimers, the pair corrections and a trained network."""
    g = _gen(seed)
    n, nt = case["monomers"], case["trimers"]
    cen = torch.rand((n, 3), dtype=F64, device=DEV, generator=g) * 12.5 * n ** (1.0 / 3.0)
    nocc = torch.randint(8, 21, (n,), device=DEV, generator=g).to(torch.int32)
    first = torch.randint(0, n, (nt,), device=DEV, generator=g)
    step = torch.randint(1, max(2, n // 2), (nt, 2), device=DEV, generator=g)
    tri = torch.stack([first, (first + step[:, 0]) % n, (first + step[:, 0] + step[:, 1]) % n], 1)
    tri = torch.sort(tri, dim=1)[0].to(torch.int32).contiguous()
    de = -(10.0 ** (torch.rand((n, n), dtype=F64, device=DEV, generator=g) * 6 - 9))
    return {"cen": cen, "nocc": nocc, "tri": tri, "de": torch.triu(de, 1) + torch.triu(de, 1).T,
            "master": _network(g),
            "mean": torch.tensor([30, 40, 50, 11, 14, 17, -7.5, -6, -4.5], dtype=torch.float32, device=DEV),
            "std": torch.tensor([12, 12, 12, 3, 3, 3, 1.2, 1.2, 1.2], dtype=torch.float32, device=DEV)}


def _full_mo(case, seed):
    """Full-MO tensor, energies, densities and J^-1/2 of the gradient step: the spread of B
    keeps the Z-vector operator positive definite, as a stable reference does."""
    o, v, x = case["nocc"], case["nvir"], case["naux"]
    n, g = o + v, _gen(seed)
    B = torch.randn((n, n, x), dtype=F64, device=DEV, generator=g) * (0.25 / (o * v * x) ** 0.25)
    B[:o, :o] = (B[:o, :o] + B[:o, :o].transpose(0, 1)) / math.sqrt(2.0)
    B[o:, o:] = (B[o:, o:] + B[o:, o:].transpose(0, 1)) / math.sqrt(2.0)
    B[o:, :o] = B[:o, o:].transpose(0, 1)
    eps = torch.cat([_uniform(g, o, -1.5, -0.3), _uniform(g, v, 0.2, 3.0)])
    gamma = torch.randn((o, v, x), dtype=F64, device=DEV, generator=g) * 1e-3
    pij = torch.randn((o, o), dtype=F64, device=DEV, generator=g) * 1e-3
    pab = torch.randn((v, v), dtype=F64, device=DEV, generator=g) * 1e-3
    j = torch.randn((x, x), dtype=F64, device=DEV, generator=g) / math.sqrt(x)
    jmh = torch.eye(x, dtype=F64, device=DEV) + 0.2 * (j + j.T)
    return B, eps, gamma, -(pij @ pij.T), pab @ pab.T, jmh


# ------------------------------------------------------------------------------ one pass

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("fragment", "batch"):
        grad = case.get("grad", True)
        opts = {} if grad else {"slices_v": 8} if case["precision"] == "bf16" else {}
        eng = rimp2.Engine(_dims(case), precision=case["precision"], want_gamma=grad, want_p=grad,
                           want_epair=grad, **opts)
        for k, f in enumerate(_fragments(case, seed)):
            o, v, x = eng.dims[k]
            b, e, _, _ = eng.offsets[k]
            eng.B[b:b + o * v * x].copy_(f.B.reshape(-1))
            eng.eps[e:e + o].copy_(f.eo)
            eng.eps[e + o:e + o + v].copy_(f.ev)
        return {"kind": kind, "eng": eng, "grad": grad}
    if kind == "assembly":
        mono, frags, coeff, off, pools = _pools(case, seed)
        asm = rimp2.MBEAssembly([m[0] for m in mono], [m[1] for m in mono], [m[2] for m in mono],
                                frags, coeff, *([a[0][k] for a in off] for k in range(3)))
        return {"kind": kind, "asm": asm, "pools": pools, "out": asm.outputs()}
    if kind == "train":
        return {"kind": kind, **_screen(case, seed)}
    if kind == "predict":
        return {"kind": kind, **_candidates(case, seed)}
    o, v, x = case["nocc"], case["nvir"], case["naux"]
    ws = torch.empty(rimp2.zvector_workspace_size(o, v, x), dtype=torch.uint8, device=DEV)
    return {"kind": kind, "args": _full_mo(case, seed), "ws": ws}


def run(s):
    kind = s["kind"]
    if kind in ("fragment", "batch"):
        e = s["eng"]
        e.run()
        out = {"energy": e.energy, "energy_os": e.energy_os, "energy_scs": e.energy_scs}
        if s["grad"]:
            out.update(gamma=e.gamma, pij=e.pij, pab=e.pab, epair=e.epair)
        return out
    if kind == "assembly":
        g, pij, pab = s["out"]
        s["asm"].run(*s["pools"], g, pij, pab)
        return {"gamma": g, "pij": pij, "pab": pab}
    if kind == "train":
        grad, loss = rimp2.mlp_grad(s["master"], s["feats"], s["y"], s["idx"], s["idx"].numel(),
                                    s["mean"], s["std"])
        s["t"] += 1
        rimp2.mlp_adam(s["master"], grad, s["m"], s["v"], s["t"], 2e-3)
        return {"grad": grad, "loss": loss, "master": s["master"], "m": s["m"], "v": s["v"]}
    if kind == "predict":
        f = rimp2.screen_features(s["cen"], s["nocc"], s["tri"], s["de"])
        return {"feats": f, "pred": rimp2.mlp_predict(s["master"], f, s["mean"], s["std"])}
    B, eps, gamma, pij, pab, jmh = s["args"]
    out = rimp2.zvector(B, eps, gamma, pij, pab, jmh=jmh, workspace=s["ws"], sync=False)
    return {k: out[k] for k in ("gamma_p", "lp", "lpp", "dai", "info")}


# ------------------------------------------------------------------------------ work

def _frag_work(o, v, x, grad):
    """FLOPs (V over the pairs i <= j, P_ab and P_ij over one triangle: all are symmetric)
    and bytes (B and the orbital energies in, the requested outputs out)."""
    flops = o * (o + 1.0) * v * v * x
    data = o * v * x + o + v + 3.0
    if grad:
        flops += 2.0 * o * o * v * v * x + 1.0 * o * o * v * v * (v + 1) + 1.0 * o * (o + 1) * o * v * v
        data += o * v * x + 2.0 * o * o + v * v
    return 8.0 * data, flops


def work(case):
    kind = case["kind"]
    if kind in ("fragment", "batch"):
        each = [_frag_work(*d, case.get("grad", True)) for d in _dims(case)]
        return {"bytes": sum(e[0] for e in each), "flops": sum(e[1] for e in each)}
    if kind == "assembly":
        mono, frags, _ = _polymers(case)
        items, blocks = 0.0, {}
        for f in frags:
            o, v, x = (sum(mono[m][k] for m in f) for k in range(3))
            items += o * v * x + o * o + v * v
            for t in itertools.product(f, f, f):
                blocks[t] = mono[t[0]][0] * mono[t[1]][1] * mono[t[2]][2]
        dense = sum(m[0] for m in mono) ** 2 + sum(m[1] for m in mono) ** 2
        return {"bytes": 8.0 * (items + sum(blocks.values()) + dense), "flops": 2.0 * items}
    net = sum(o * i for o, i in _LAYERS)
    if kind == "train":
        return {"bytes": 4.0 * (11 * case["batch"] + 8 * rimp2.MLP_PARAMS), "flops": 6.0 * net * case["batch"]}
    if kind == "predict":
        n = case["trimers"]
        return {"bytes": 4.0 * 13 * n + 8.0 * case["monomers"] ** 2, "flops": 2.0 * net * n}
    o, v, x = case["nocc"], case["nvir"], case["naux"]
    n = o + v
    # Gamma^P, L' and L'', the right-hand side, and ten iterations (a common count) of the
    # exchange product
    flops = 2.0 * o * v * x * x + 4.0 * o * n * v * x + 2.0 * o ** 3 * x + 2.0 * o * o * v * x + \
        4.0 * o * v * v * x + 10 * 4.0 * o * o * v * x
    return {"bytes": 8.0 * (n * n * x + 2 * o * v * x + x * x), "flops": flops}


# ------------------------------------------------------------------------------ 64-bit results

def _exact_fragment(f, grad):
    o, v, x = f.B.shape
    B = f.B.reshape(o * v, x)
    gamma = torch.empty_like(f.B)
    pij = torch.zeros((o, o), dtype=F64, device=DEV)
    pab = torch.zeros((v, v), dtype=F64, device=DEV)
    ep = torch.empty((o, o), dtype=F64, device=DEV)
    eos = torch.empty((o, o), dtype=F64, device=DEV)
    for i in range(o):                                   # rows (i, a) of the pair blocks
        V = (f.B[i] @ B.T).view(v, o, v)                 # [a][j][b]
        T = V / (f.eo[i] + f.eo[None, :, None] - f.ev[:, None, None] - f.ev[None, None, :])
        Tt = 2.0 * T - T.transpose(0, 2)
        ep[i] = (Tt * V).sum((0, 2))
        eos[i] = (T * V).sum((0, 2))
        if grad:
            gamma[i] = Tt.reshape(v, o * v) @ B
            pab += Tt.reshape(v, o * v) @ T.reshape(v, o * v).T
            # P_jk = -sum Tt_ij(a,b) T_ik(a,b): the pair symmetry T_ij(a,b) = T_ji(b,a)
            pij -= Tt.transpose(0, 1).reshape(o, v * v) @ T.transpose(0, 1).reshape(o, v * v).T
    e, os_ = ep.sum(), eos.sum()
    return {"energy": e, "energy_os": os_, "energy_scs": 1.2 * os_ + (e - os_) / 3.0,
            "gamma": gamma, "pij": pij, "pab": pab, "epair": ep}


def _exact_assembly(case, seed):
    mono, frags, coeff, off, (gp, ip, ap) = _pools(case, seed)
    blocks = {}
    for f in frags:
        for t in itertools.product(f, f, f):
            blocks[t] = mono[t[0]][0] * mono[t[1]][1] * mono[t[2]][2]
    start, at = {}, 0
    for t in sorted(blocks):                             # blocks in (I, J, K) order
        start[t] = at
        at += blocks[t]
    run0 = [[0] + list(itertools.accumulate(m[k] for m in mono)) for k in range(3)]
    G = torch.zeros(max(at, 1), dtype=F64, device=DEV)
    O = torch.zeros((run0[0][-1],) * 2, dtype=F64, device=DEV)
    V = torch.zeros((run0[1][-1],) * 2, dtype=F64, device=DEV)
    for f, c, (b, (o, v, x)) in zip(frags, coeff, off):
        g = gp[b[0]:b[0] + o * v * x].view(o, v, x)
        p, q = ip[b[1]:b[1] + o * o].view(o, o), ap[b[2]:b[2] + v * v].view(v, v)
        r = [[0] + list(itertools.accumulate(mono[m][k] for m in f)) for k in range(3)]
        for a, I in enumerate(f):
            for d, J in enumerate(f):
                O[run0[0][I]:run0[0][I + 1], run0[0][J]:run0[0][J + 1]] += c * p[r[0][a]:r[0][a + 1], r[0][d]:r[0][d + 1]]
                V[run0[1][I]:run0[1][I + 1], run0[1][J]:run0[1][J + 1]] += c * q[r[1][a]:r[1][a + 1], r[1][d]:r[1][d + 1]]
                for e, K in enumerate(f):
                    s = start[(I, J, K)]
                    blk = g[r[0][a]:r[0][a + 1], r[1][d]:r[1][d + 1], r[2][e]:r[2][e + 1]]
                    G[s:s + blocks[(I, J, K)]] += c * blk.reshape(-1)
    return {"gamma": G, "pij": O, "pab": V}


def _forward(theta, x):
    """The 9-64-64-64-1 SiLU network in 64 bits."""
    at = 0
    for k, (o, i) in enumerate(_LAYERS):
        W, b = theta[at:at + o * i].view(o, i), theta[at + o * i:at + o * i + o]
        at += o * i + o
        x = x @ W.T + b
        if k < 3:
            x = x * torch.sigmoid(x)
    return x[:, 0]


def _rounded(master):
    """The weights as the network uses them: rounded to BF16, here held in 64 bits."""
    return master.to(torch.bfloat16).to(F64)


def _exact_train(case, seed):
    s = _screen(case, seed)
    rows = s["idx"].long()
    theta = _rounded(s["master"]).requires_grad_(True)
    x = (s["feats"][rows].to(F64) - s["mean"].to(F64)) / s["std"].to(F64)
    loss = (_forward(theta, x) - s["y"][rows].to(F64)).square().mean()
    grad, = torch.autograd.grad(loss, theta)
    t = s["t"] + 1
    m = 0.9 * s["m"].to(F64) + 0.1 * grad
    v = 0.999 * s["v"].to(F64) + 0.001 * grad * grad
    w = s["master"].to(F64) - 2e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"grad": grad, "loss": loss.detach().reshape(1), "master": w, "m": m, "v": v}


def _exact_predict(case, seed):
    s = _candidates(case, seed)
    t = s["tri"].long()
    pairs = ((0, 1), (0, 2), (1, 2))
    d = torch.stack([(s["cen"][t[:, a]] - s["cen"][t[:, b]]).norm(dim=1) for a, b in pairs], 1)
    n = s["nocc"][t].to(F64)
    e = torch.stack([(s["de"][t[:, a], t[:, b]].abs() + 1e-16).log10() for a, b in pairs], 1)
    f = torch.cat([torch.sort(k, dim=1)[0] for k in (d, n, e)], 1)
    return {"feats": f, "pred": _forward(_rounded(s["master"]), (f - s["mean"].to(F64)) / s["std"].to(F64))}


def _exact_gradient(case, seed):
    B, eps, gamma, pij, pab, jmh = _full_mo(case, seed)
    o, v, x = gamma.shape
    n = o + v
    Bov, Boo, Bvv = B[:o, o:], B[:o, :o], B[o:, o:]
    gv, go = gamma.reshape(o, v * x), gamma.transpose(0, 1).reshape(v, o * x)
    lp = gv @ B[:, o:].reshape(n, v * x).T                       # sum_aQ Gamma^Q_ia B^Q_qa
    lpp = go @ B[:o].transpose(0, 1).reshape(n, o * x).T         # sum_iQ Gamma^Q_ia B^Q_iq
    de = (Boo * pij[:, :, None]).sum((0, 1)) + (Bvv * pab[:, :, None]).sum((0, 1))
    rhs = lpp[:, :o].T - lp[:, o:] - 2.0 * (Bov @ de)
    U = torch.einsum("kl,ikq->ilq", pij, Boo)
    rhs = rhs + U.reshape(o, o * x) @ Bov.transpose(0, 1).reshape(v, o * x).T
    W = torch.einsum("bc,ibq->icq", pab, Bov)
    rhs = rhs + W.reshape(o, v * x) @ Bvv.reshape(v, v * x).T
    A = (Bov.reshape(o * v, x) @ Bov.reshape(o * v, x).T).view(o, v, o, v)   # (ia|jb)
    A = (2.0 * A - A.transpose(0, 2)).reshape(o * v, o * v)
    A.diagonal().add_(0.5 * (eps[None, o:] - eps[:o, None]).reshape(-1))
    dai = torch.linalg.solve(A, rhs.reshape(-1)).view(o, v)
    return {"gamma_p": gamma @ jmh.T, "lp": lp, "lpp": lpp, "dai": dai, "info": None}


def exact(case, seed):
    """What `run` returns for these inputs, in 64 bits, by plain torch (the split-path
    fragments take the same formulas; the iteration record of the Z-vector has no such
    value)."""
    kind = case["kind"]
    if kind in ("fragment", "batch"):
        grad = case.get("grad", True)
        each = [_exact_fragment(f, grad) for f in _fragments(case, seed)]
        out = {k: torch.stack([e[k] for e in each]) for k in ("energy", "energy_os", "energy_scs")}
        if grad:
            out.update({k: torch.cat([e[k].reshape(-1) for e in each]) for k in ("gamma", "pij", "pab", "epair")})
        return out
    return {"assembly": _exact_assembly, "train": _exact_train, "predict": _exact_predict,
            "gradient": _exact_gradient}[kind](case, seed)
