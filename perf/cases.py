"""Timing cases: the work that a user of the library has it do, through its Python binding.

A two-site DMRG program (Sec. 11 of arXiv 2401.01921) spends its time in five calls: one application
of the effective Hamiltonian (``Network.launch_into``), the Lanczos solve built on it (``lanczos``),
the truncated SVD of the result (``svd_truncate``), the environment update (another network) and,
when many small problems run side by side, the batched apply (``Batch.launch_into``).  Every case is one
pass of one of them, and the last listed one is a whole bond update with new networks.

Inputs are made on the GPU from the seed alone: N(0, 1) blocks, environments symmetrised so that the
effective Hamiltonian is Hermitian (as in DMRG), optionally scaled over three decades by charge sector,
wavefunctions for the SVD with a spectrum that falls off exponentially.  Sector lists, MPO tensors and
blueprints are the ones of ``tnx_inputs``.
"""
import functools
import itertools
import math
import random

import numpy as np
import torch

import paper_2401_01921_gb300 as tnx
import tnx_inputs as I
from paper_2401_01921_gb300.heff import make_bonds

DEV = "cuda"
PRODUCT_SPEC = "U: a, s1, k\nS: k, l\nV: l, s2, b\nTOUT: a, s1, s2, b\nORDER:\n"


def _nsec(chi):
    """Number of charge steps of a Heisenberg bond of dimension chi (20 at 512, 40 at 2048)."""
    return max(4, int(round(20 * (chi / 512) ** 0.5)))


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest solve of the benchmark (no charges, bond dimension 32): launches and latency
        {"name": "solve_dense_32", "kind": "solve", "model": "dense", "chi": 32, "scaled": False, "steps": 20,
         "prec": "split_bf16"},
        # a solve early in a sweep, in the precision that a network has by default
        {"name": "solve_heis_150_f64", "kind": "solve", "model": "heisenberg", "chi": 150, "scaled": False, "steps": 20,
         "prec": "f64"},
        # an ordinary solve of a DMRG sweep
        {"name": "solve_heis_512", "kind": "solve", "model": "heisenberg", "chi": 512, "scaled": False, "steps": 20,
         "prec": "split_bf16"},
        # the benchmark's headline: a large solve, sectors scaled over three decades
        {"name": "solve_heis_2048", "kind": "solve", "model": "heisenberg", "chi": 2048, "scaled": True, "steps": 20,
         "prec": "split_bf16"},
        # one served apply at a ragged, odd bond dimension
        {"name": "apply_heis_777", "kind": "apply", "model": "heisenberg", "chi": 777, "scaled": False,
         "prec": "split_bf16"},
        # one apply at the largest bond dimension of the benchmark
        {"name": "apply_heis_4096", "kind": "apply", "model": "heisenberg", "chi": 4096, "scaled": True,
         "prec": "split_bf16"},
        # two charges, four local states: many small ragged blocks
        {"name": "apply_hubbard_601", "kind": "apply", "model": "hubbard", "chi": 601, "scaled": False,
         "prec": "split_bf16"},
        # independent small problems side by side (a parameter scan)
        {"name": "batch_hubbard_48", "kind": "batch", "count": 48, "lo": 6.0, "hi": 10.0, "prec": "split_bf16"},
        # the environment update of a sweep
        {"name": "env_heis_2048", "kind": "env", "chi": 2048, "prec": "split_bf16"},
        # truncation of a two-site wavefunction early in a sweep
        {"name": "svd_heis_200", "kind": "svd", "chi": 200, "decades": 12.0},
        # the same at the bond dimension where a sweep spends most of its time on it
        {"name": "svd_heis_1024", "kind": "svd", "chi": 1024, "decades": 12.0},
        # a whole bond update as a sweep does it: new networks, solve, truncation, new wavefunction
        {"name": "bond_heis_256", "kind": "bond", "chi": 256, "steps": 12, "prec": "split_bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "apply", "apply", "batch", "env", "svd", "svd", "bond"])
    prec = rng.choice(["split_bf16", "split_bf16", "split_f16", "f64"])
    if kind in ("solve", "apply"):
        model = rng.choice(["heisenberg", "heisenberg", "heisenberg", "hubbard", "dense"])
        top = {"heisenberg": 2048 if kind == "solve" else 4096, "hubbard": 700, "dense": 64}[model]
        if prec == "f64":
            top = min(top, 500)
        case = {"kind": kind, "model": model, "chi": _log(rng, 24 if model == "dense" else 40, top),
                "scaled": model == "heisenberg" and rng.random() < 0.5}
        if kind == "solve":
            case["steps"] = rng.randint(5, 20)
    elif kind == "batch":
        lo = rng.uniform(5.5, 7.0)
        case = {"kind": kind, "count": rng.randint(5, 40), "lo": lo, "hi": rng.uniform(lo + 1.0, 9.5)}
    elif kind == "env":
        case = {"kind": kind, "chi": _log(rng, 60, 2048 if prec != "f64" else 500)}
    elif kind == "svd":
        return {"kind": kind, "chi": _log(rng, 40, 900), "decades": rng.uniform(6.0, 14.0)}
    else:
        case = {"kind": kind, "chi": _log(rng, 50, 256), "steps": rng.randint(6, 12)}
    case["prec"] = prec
    return case


# ------------------------------------------------------------------ block structure (plain Python)
def _workload(case):
    model, chi = case.get("model", "heisenberg"), case["chi"]
    if model == "dense":
        return I.dense_workload(chi)
    if model == "hubbard":
        return I.hubbard_workload(chi)
    return I.heisenberg_workload(chi, _nsec(chi))


def _batch_workloads(case):
    return [I.hubbard_workload(c) for c in I.batched_hubbard_chis(case["count"], 6, case["lo"], case["hi"])]


def _blocks(legs):
    """Sector indices of the stored (zero-flux) blocks in lexicographic order, with their shapes."""
    return _blocks_of(tuple((d, tuple(s)) for d, s in legs))


@functools.lru_cache(maxsize=512)
def _blocks_of(legs):
    *head, (last_dir, last) = legs
    at = {}
    for i, (q, _) in enumerate(last):
        at.setdefault(tuple(-last_dir * x for x in q), []).append(i)
    out = []
    for idx in itertools.product(*[range(len(s)) for _, s in head]):
        flux = tuple(sum(d * s[i][0][c] for (d, s), i in zip(head, idx)) for c in range(len(last[0][0])))
        for i in at.get(flux, ()):
            qn = idx + (i,)
            out.append((qn, tuple(s[k][1] for (_, s), k in zip(legs, qn))))
    return out


def _size(legs):
    return sum(math.prod(sh) for _, sh in _blocks(legs))


def _split(flat, legs):
    """{sector indices: block}, the blocks being views of the flat buffer."""
    out, o = {}, 0
    for qn, sh in _blocks(legs):
        n = math.prod(sh)
        out[qn] = flat[o:o + n].view(sh)
        o += n
    return out


def _mpo(legs, Wg):
    off = [np.concatenate([[0], np.cumsum([d for _, d in s])]) for _, s in legs]
    flat = [Wg[tuple(slice(o[k], o[k] + d) for o, k, d in zip(off, qn, sh))].reshape(-1) for qn, sh in _blocks(legs)]
    return torch.from_numpy(np.concatenate(flat)).to(DEV)


def _env_bar(wl):
    """Position of the adjoint channel of every MPO channel (S+ <-> S-, c <-> c+), in grouped order."""
    bar = [0, 2, 1, 4, 3, 5] if wl.kind == "hubbard" else I.channel_bar_heisenberg(wl.mpo.W.shape[0])
    pos = wl.mpo.channel_pos
    out = [0] * len(pos)
    for ch, p in enumerate(pos):
        out[p] = pos[bar[ch]]
    return out


def _randn(n, g):
    return torch.randn(n, generator=g, device=DEV, dtype=torch.float64)


def _heff_values(wl, g, rnd, symmetric, scaled):
    """Flat buffers of L, psi, W1, W2, R."""
    legs = I.heff_bonds(wl)
    T = {n: _randn(_size(legs[n]), g) for n in ("L", "psi", "R")}
    for n in ("W1", "W2"):
        T[n] = _mpo(legs[n], wl.mpo.W_grouped())
    if symmetric:
        bar = _env_bar(wl)
        for n in ("L", "R"):
            wsec = legs[n][1][1]
            where = [(k, i) for k, (_, d) in enumerate(wsec) for i in range(d)]
            first = [where.index((k, 0)) for k in range(len(wsec))]
            src, dst = _split(T[n], legs[n]), torch.empty_like(T[n])
            for (a, w, b), blk in _split(dst, legs[n]).items():
                for i in range(blk.shape[1]):
                    w2, i2 = where[bar[first[w] + i]]
                    torch.add(src[a, w, b][:, i, :], src[b, w2, a][:, i2, :].T, out=blk[:, i, :])
            T[n] = dst.mul_(0.5)
    if scaled:
        u = {n: [rnd.random() for _ in range(len(legs[n][0][1]))] for n in ("L", "psi", "R")}
        for n in ("L", "psi", "R"):
            for qn, blk in _split(T[n], legs[n]).items():
                blk.mul_(10.0 ** (-3.0 * u[n][qn[0]] if n == "psi" else -1.5 * (u[n][qn[0]] + u[n][qn[2]])))
    return legs, T


def _env_values(case, g):
    legs = I.env_bonds(case["chi"], _nsec(case["chi"]))
    T = {n: _randn(_size(legs[n]), g) for n in ("L", "A")}
    T["W"] = _mpo(legs["W"], I.heisenberg_mpo().W_grouped())
    T["Ad"] = T["A"].clone()
    legs["Ad"] = [(-d, s) for d, s in legs["A"]]
    return legs, T


def _charge_blocks(legs):
    """The matrix blocks of a two-site wavefunction: {row charge: (rows {(a, s1): (offset, dim)}, columns)}."""
    out = {}
    for qn, sh in _blocks(legs):
        key = tuple(x + y for x, y in zip(legs[0][1][qn[0]][0], legs[1][1][qn[1]][0]))
        rows, cols = out.setdefault(key, ({}, {}))
        rows.setdefault(qn[:2], sh[0] * sh[1])
        cols.setdefault(qn[2:], sh[2] * sh[3])
    for key, sides in out.items():
        placed = []
        for s in sides:
            o, t = 0, {}
            for k in sorted(s):
                t[k] = (o, s[k])
                o += s[k]
            placed.append(t)
        out[key] = placed
    return out


def _dim(side):
    return sum(d for _, d in side.values())


def _theta_values(case, g):
    """A normalised two-site wavefunction whose charge blocks have spectra falling over `decades`."""
    legs = I.heff_bonds(_workload(case))["psi"]
    flat = torch.zeros(_size(legs), dtype=torch.float64, device=DEV)
    views = _split(flat, legs)
    for rows, cols in _charge_blocks(legs).values():
        m, n = _dim(rows), _dim(cols)
        c = min(m, n)
        fall = 10.0 ** (-case["decades"] * torch.arange(c, device=DEV, dtype=torch.float64) / c)
        M = (_randn(m * c, g).view(m, c) * fall) @ _randn(c * n, g).view(c, n) / c
        for rk, (r0, rd) in rows.items():
            for ck, (c0, cd) in cols.items():
                blk = views[rk + ck]
                blk.copy_(M[r0:r0 + rd, c0:c0 + cd].reshape(blk.shape))
    return legs, flat.div_(torch.linalg.vector_norm(flat))


# ------------------------------------------------------------------ inputs on the GPU
class _Buffer:
    """A tensor's device buffer for torch (no copy)."""

    def __init__(self, t):
        self.__cuda_array_interface__ = {"shape": (t.nelem,), "typestr": "<f8", "data": (t.data_ptr, False),
                                         "version": 3, "strides": None}


def _view(t):
    if t.nelem == 0:
        return torch.zeros(0, dtype=torch.float64, device=DEV)
    return torch.as_tensor(_Buffer(t), device=DEV)


_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = tnx.Context(torch.cuda.current_device())
    return _ctx


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _tensor(ctx, legs, flat, nsym):
    t = tnx.Tensor(ctx, make_bonds(ctx, legs, nsym))
    if t.nelem:
        _view(t).copy_(flat)
    return t


def _network(ctx, spec, T, order, prec):
    net = tnx.Network(ctx, spec)
    for name, t in T.items():
        net.put(name, t)
    if order in (True, "sparse"):
        net.set_order(order)
    else:
        net.set_order(False, order)
    net.set_precision(prec)
    return net


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    with torch.cuda.stream(ctx.stream):
        g, rnd = _generator(seed), random.Random(seed)
        st = {"case": case, "ctx": ctx}
        if kind in ("solve", "apply", "bond"):
            wl = _workload(case)
            legs, V = _heff_values(wl, g, rnd, kind != "apply", case.get("scaled", False))
            st["T"] = T = {n: _tensor(ctx, legs[n], V[n], wl.nsym) for n in I.HEFF_NAMES}
            if kind != "bond":
                st["net"] = _network(ctx, I.HEFF_SPEC, T, "sparse", case["prec"])
                st["out"] = tnx.Tensor(ctx, T["psi"].bonds)
        elif kind == "env":
            legs, V = _env_values(case, g)
            st["T"] = T = {n: _tensor(ctx, legs[n], V[n], 1) for n in ("L", "A", "W", "Ad")}
            st["net"] = _network(ctx, I.ENV_LEFT_SPEC, T, "sparse", case["prec"])
            st["out"] = tnx.Tensor(ctx, [T["A"].bonds[2], T["W"].bonds[3], T["Ad"].bonds[2]])
        elif kind == "svd":
            legs, flat = _theta_values(case, g)
            st["theta"] = _tensor(ctx, legs, flat, 1)
        elif kind == "batch":
            st["T"], st["nets"], st["out"] = [], [], []
            for wl in _batch_workloads(case):
                legs, V = _heff_values(wl, g, rnd, False, False)
                T = {n: _tensor(ctx, legs[n], V[n], wl.nsym) for n in I.HEFF_NAMES}
                st["T"].append(T)
                # L as the right operand: the order that the library's benchmark runs batches in
                st["nets"].append(_network(ctx, I.HEFF_SPEC, T, "(((psi,R),(W1,W2)),L)", case["prec"]))
                st["out"].append(tnx.Tensor(ctx, T["psi"].bonds))
            st["batch"] = tnx.Batch(ctx, st["nets"])
    ctx.stream.synchronize()
    return st


def _truncate(st, theta, keep):
    """theta cut to `keep` values: the new wavefunction U S V, which does not depend on the vectors' signs (the
    factors' own shapes depend on which charges the kept values fall to), and what was dropped."""
    U, S, V, largest, weight = tnx.svd_truncate(theta, 2, keep)
    net = _network(st["ctx"], PRODUCT_SPEC, {"U": U, "S": S, "V": V}, True, "f64")
    new = net.launch(theta.bonds)
    st["kept"] = (U, S, V, net, new)   # the outputs live in these buffers until the next pass
    return {"theta": _view(new), "largest_dropped": largest, "dropped_weight": weight}


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind in ("apply", "env"):
        st["net"].launch_into(st["out"])
        return _view(st["out"])
    if kind == "solve":
        value, _ = tnx.lanczos(st["net"], "psi", st["T"]["psi"], case["steps"], st["out"])
        return {"value": value, "vector": _view(st["out"])}
    if kind == "batch":
        st["batch"].launch_into(st["out"])
        return [_view(o) for o in st["out"]]
    if kind == "svd":
        return _truncate(st, st["theta"], case["chi"])
    st["evec"] = vec = tnx.Tensor(st["ctx"], st["T"]["psi"].bonds)
    st["net"] = net = _network(st["ctx"], I.HEFF_SPEC, st["T"], "sparse", case["prec"])
    value, _ = tnx.lanczos(net, "psi", st["T"]["psi"], case["steps"], vec)
    return {"value": value, "vector": _view(vec), **_truncate(st, vec, case["chi"])}


# ------------------------------------------------------------------ work
def _pair(A, la, B, lb):
    """Matched block pairs of two operands given as {sector indices: shape}: the product's labels, its
    blocks and the flops 2 m k n."""
    common = [x for x in la if x in lb]
    fb = [i for i, x in enumerate(lb) if x not in common]
    fa = [i for i, x in enumerate(la) if x not in common]
    ka, kb = [la.index(x) for x in common], [lb.index(x) for x in common]
    by = {}
    for q, sh in B.items():
        by.setdefault(tuple(q[i] for i in kb), []).append((tuple(q[i] for i in fb), tuple(sh[i] for i in fb)))
    out, flops = {}, 0
    for q, sh in A.items():
        for qb, sb in by.get(tuple(q[i] for i in ka), ()):
            out[tuple(q[i] for i in fa) + qb] = tuple(sh[i] for i in fa) + sb
            flops += 2 * math.prod(sh) * math.prod(sb)
    return out, [la[i] for i in fa] + [lb[i] for i in fb], flops


HEFF_LABELS = {"L": ["a", "w0", "ap"], "psi": ["a", "s1", "s2", "b"], "W1": ["w0", "s1p", "s1", "w1"],
               "W2": ["w1", "s2p", "s2", "w2"], "R": ["b", "w2", "bp"]}
ENV_LABELS = {"L": ["a", "w", "ap"], "A": ["a", "s", "b"], "W": ["w", "sp", "s", "wp"], "Ad": ["ap", "sp", "bp"]}


def _heff_work(wl):
    """(flops of one apply, elements of the inputs, elements of psi)."""
    legs = I.heff_bonds(wl)
    S = {n: dict(_blocks(legs[n])) for n in legs}
    X, lx, f1 = _pair(S["psi"], HEFF_LABELS["psi"], S["R"], HEFF_LABELS["R"])
    W, lw, f2 = _pair(S["W1"], HEFF_LABELS["W1"], S["W2"], HEFF_LABELS["W2"])
    Y, ly, f3 = _pair(X, lx, W, lw)
    _, _, f4 = _pair(Y, ly, S["L"], HEFF_LABELS["L"])
    n = {k: sum(math.prod(s) for s in S[k].values()) for k in S}
    return f1 + f2 + f3 + f4, sum(n.values()), n["psi"]


def _svd_work(case):
    legs = I.heff_bonds(_workload(case))["psi"]
    flops = 0
    for rows, cols in _charge_blocks(legs).values():
        m, n = _dim(rows), _dim(cols)
        c = min(m, n)
        flops += 4 * m * n * c          # the reduction to bidiagonal form, which every method exceeds
    # theta in, the new wavefunction out
    return {"bytes": 16 * _size(legs), "flops": flops}


def work(case):
    kind = case["kind"]
    if kind in ("apply", "solve", "bond"):
        f, nin, n = _heff_work(_workload(case))
        k = case.get("steps", 1)
        # a Lanczos step adds a dot product, the three-term step and a norm
        w = {"bytes": 8 * (nin + n), "flops": k * f + (8 * k * n if kind != "apply" else 0)}
        if kind == "bond":
            s = _svd_work(case)
            w = {x: w[x] + s[x] for x in w}
        return w
    if kind == "batch":
        ws = [_heff_work(wl) for wl in _batch_workloads(case)]
        return {"bytes": 8 * sum(nin + n for _, nin, n in ws), "flops": sum(f for f, _, _ in ws)}
    if kind == "svd":
        return _svd_work(case)
    legs = I.env_bonds(case["chi"], _nsec(case["chi"]))
    legs["Ad"] = [(-d, s) for d, s in legs["A"]]
    S = {n: dict(_blocks(legs[n])) for n in legs}
    X, lx, f1 = _pair(S["L"], ENV_LABELS["L"], S["A"], ENV_LABELS["A"])
    Y, ly, f2 = _pair(X, lx, S["W"], ENV_LABELS["W"])
    Z, _, f3 = _pair(Y, ly, S["Ad"], ENV_LABELS["Ad"])
    n = {k: sum(math.prod(s) for s in S[k].values()) for k in S}
    return {"bytes": 8 * (n["L"] + n["A"] + n["W"] + sum(math.prod(s) for s in Z.values())), "flops": f1 + f2 + f3}


# ------------------------------------------------------------------ the same results in plain torch FP64
def _mul(A, la, B, lb):
    """Block-sparse product of {sector indices: block} operands over their common labels."""
    common = [x for x in la if x in lb]
    ka, kb = [la.index(x) for x in common], [lb.index(x) for x in common]
    fa = [i for i in range(len(la)) if i not in ka]
    fb = [i for i in range(len(lb)) if i not in kb]
    by = {}
    for q, blk in B.items():
        by.setdefault(tuple(q[i] for i in kb), []).append((tuple(q[i] for i in fb), blk))
    out = {}
    for q, blk in A.items():
        for qb, bb in by.get(tuple(q[i] for i in ka), ()):
            key = tuple(q[i] for i in fa) + qb
            p = torch.tensordot(blk, bb, (ka, kb))
            out[key] = out[key].add_(p) if key in out else p
    return out, [la[i] for i in fa] + [lb[i] for i in fb]


def _lay_out(Z, lz, labels, legs):
    perm = [lz.index(x) for x in labels]
    flat = torch.zeros(_size(legs), dtype=torch.float64, device=DEV)
    views = _split(flat, legs)
    for q, blk in Z.items():
        views[tuple(q[i] for i in perm)].copy_(blk.permute(perm))
    return flat


def _heff_apply(legs, V):
    """flat psi -> flat H psi."""
    S = {n: _split(V[n], legs[n]) for n in ("L", "W1", "W2", "R")}
    W, lw = _mul(S["W1"], HEFF_LABELS["W1"], S["W2"], HEFF_LABELS["W2"])

    def apply(x):
        X, lx = _mul(_split(x, legs["psi"]), HEFF_LABELS["psi"], S["R"], HEFF_LABELS["R"])
        Y, ly = _mul(X, lx, W, lw)
        Z, lz = _mul(Y, ly, S["L"], HEFF_LABELS["L"])
        return _lay_out(Z, lz, ["ap", "s1p", "s2p", "bp"], legs["psi"])

    return apply


def _exact_lanczos(apply, v0, steps):
    v = v0 / torch.linalg.vector_norm(v0)
    basis, alpha, beta = [v], [], []
    for j in range(steps):
        w = apply(basis[j])
        alpha.append(torch.dot(basis[j], w).item())
        for _ in range(2):
            Vm = torch.stack(basis)
            w = w - Vm.T @ (Vm @ w)
        b = torch.linalg.vector_norm(w).item()
        if j + 1 == steps or b < 1e-14 * max([abs(a) for a in alpha] + beta):
            break
        beta.append(b)
        basis.append(w / b)
    lam, y = np.linalg.eigh(np.diag(alpha) + np.diag(beta[:len(alpha) - 1], 1) + np.diag(beta[:len(alpha) - 1], -1))
    y = y[:, 0] * np.sign(y[np.argmax(np.abs(y[:, 0])), 0])
    return float(lam[0]), torch.stack(basis).T @ torch.from_numpy(y).to(DEV)


def _exact_truncate(legs, flat, keep):
    views = _split(flat, legs)
    parts, values = [], []
    groups = sorted(_charge_blocks(legs).items())
    for i, (_, (rows, cols)) in enumerate(groups):
        M = torch.zeros(_dim(rows), _dim(cols), dtype=torch.float64, device=DEV)
        for rk, (r0, rd) in rows.items():
            for ck, (c0, cd) in cols.items():
                M[r0:r0 + rd, c0:c0 + cd] = views[rk + ck].reshape(rd, cd)
        u, s, v = (x.to(DEV) for x in torch.linalg.svd(M.cpu(), full_matrices=False))
        parts.append((rows, cols, u, s, v))
        values += [(x, i) for x in s.tolist()]
    values.sort(key=lambda t: -t[0])
    kept = [0] * len(groups)
    for _, i in values[:keep]:
        kept[i] += 1
    new = torch.zeros_like(flat)
    out = _split(new, legs)
    for (rows, cols, u, s, v), k in zip(parts, kept):
        M = (u[:, :k] * s[:k]) @ v[:k]
        for rk, (r0, rd) in rows.items():
            for ck, (c0, cd) in cols.items():
                blk = out[rk + ck]
                blk.copy_(M[r0:r0 + rd, c0:c0 + cd].reshape(blk.shape))
    rest = [x for x, _ in values[keep:]]
    return {"theta": new, "largest_dropped": rest[0] if rest else 0.0,
            "dropped_weight": math.fsum(x * x for x in rest)}


def exact(case, seed):
    g, rnd, kind = _generator(seed), random.Random(seed), case["kind"]
    if kind in ("apply", "solve", "bond"):
        wl = _workload(case)
        legs, V = _heff_values(wl, g, rnd, kind != "apply", case.get("scaled", False))
        apply = _heff_apply(legs, V)
        if kind == "apply":
            return apply(V["psi"])
        value, vec = _exact_lanczos(apply, V["psi"], case["steps"])
        out = {"value": value, "vector": vec}
        return out if kind == "solve" else {**out, **_exact_truncate(legs["psi"], vec, case["chi"])}
    if kind == "batch":
        out = []
        for wl in _batch_workloads(case):
            legs, V = _heff_values(wl, g, rnd, False, False)
            # the block loop of the larger instances would take too long
            out.append(_heff_apply(legs, V)(V["psi"]) if wl.chi <= 128 else None)
        return out
    if kind == "svd":
        legs, flat = _theta_values(case, g)
        return _exact_truncate(legs, flat, case["chi"])
    legs, V = _env_values(case, g)
    S = {n: _split(V[n], legs[n]) for n in ENV_LABELS}
    X, lx = _mul(S["L"], ENV_LABELS["L"], S["A"], ENV_LABELS["A"])
    Y, ly = _mul(X, lx, S["W"], ENV_LABELS["W"])
    Z, lz = _mul(Y, ly, S["Ad"], ENV_LABELS["Ad"])
    return _lay_out(Z, lz, ["b", "wp", "bp"], [(legs["A"][2][0], legs["A"][2][1]), legs["W"][3], legs["Ad"][2]])
