"""The work that a user of this library has it do, as cases that can be timed and compared.

A case names one call (or, for the energy's gradient, a forward and a backward pass) with its bond dimensions and
its arithmetic.  Sizes are those of the paper's range and of this repository's own runs: chi = 4 .. 16 in binary64
(the default arithmetic of every entry point), up to chi = 32 in the tensor-core modes.  `exact` repeats the call in
64 bits with plain torch contractions.
"""
import math

import numpy as np
import torch

import mera_inputs as M
import paper_1906_12030_gb300 as G
from paper_1906_12030_gb300 import autograd as A

MAPS = {"ascend": G.OP_ASCEND, "descend": G.OP_DESCEND, "env_u": G.OP_ENV_U, "env_w": G.OP_ENV_W}
# the contractions' rates (flop/s) by which drawn cases are kept below the largest listed one
RATE = {"f64": 1.2e12, "tf32": 3.5e14, "bf16": 6e14, "bf16x3": 3.2e14, "bf16x6": 1.9e14, "oz3": 1.1e14, "oz4": 9e13}
N_LAYERS, N_POW = 3, 20  # tau* = 3 and 20 power steps for rho* per sweep


def listed():
    return [
        # one ascending map at the smallest bond dimension, from a caller that owns all device memory: latency
        {"name": "ascend noalloc f64 4", "kind": "noalloc", "prec": "f64", "chi_b": 4, "chi_t": 4},
        # the first transitional layer of every sweep with chi >= 16: blocked spins (4) up to 16
        {"name": "descend f64 4-16", "kind": "descend", "prec": "f64", "chi_b": 4, "chi_t": 16},
        # energy and its four gradients, as a gradient-based optimiser asks for them; an odd bond dimension
        {"name": "energy grad f64 9", "kind": "energy_grad", "prec": "f64", "chi_b": 9, "chi_t": 9},
        # isometry environment in the middle of the paper's range, default arithmetic
        {"name": "env_w f64 10", "kind": "env_w", "prec": "f64", "chi_b": 10, "chi_t": 10},
        # the map that the rho* iteration repeats, at the paper's largest bond dimension, default arithmetic
        {"name": "descend f64 16", "kind": "descend", "prec": "f64", "chi_b": 16, "chi_t": 16},
        # polar update of a disentangler at chi = 16: one per layer and sweep, in every arithmetic
        {"name": "polar 256x256", "kind": "polar", "prec": "f64", "chi_b": 16, "n": 256, "kappa": 1e3},
        # a whole sweep in the default arithmetic, recorded once and replayed: an optimisation loop's step
        {"name": "sweep f64 8 graph", "kind": "sweep", "prec": "f64", "chi_t": 8, "graph": True},
        # a whole sweep of direct calls in the fast tensor-core mode
        {"name": "sweep bf16x3 12", "kind": "sweep", "prec": "bf16x3", "chi_t": 12, "graph": False},
        # the rho* iteration of a sweep at the paper's largest bond dimension: most of a sweep's work
        {"name": "fixed point bf16x3 16", "kind": "fixed_point", "prec": "bf16x3", "chi_b": 16, "chi_t": 16},
        # isometry environment in the accurate tensor-core mode
        {"name": "env_w oz4 16", "kind": "env_w", "prec": "oz4", "chi_b": 16, "chi_t": 16},
        # disentangler environment above the paper's range, single-plane operands
        {"name": "env_u tf32 24", "kind": "env_u", "prec": "tf32", "chi_b": 24, "chi_t": 24},
        # the largest: one ascending map at chi = 32, its rank-7 intermediates cut into slices
        {"name": "ascend bf16x3 32", "kind": "ascend", "prec": "bf16x3", "chi_b": 32, "chi_t": 32},
    ]


def _seconds(case):
    """Rough cost of a case's contractions (used to bound drawn cases)."""
    return work(case)["flops"] / RATE[case["prec"]]


def draw(rng):
    cap = 0.8 * _seconds(listed()[-1])
    while True:
        kind = rng.choice(["ascend", "descend", "env_u", "env_w", "energy_grad", "fixed_point", "polar", "sweep"])
        if kind == "polar":  # environments of u (n = chi^2) and of w (n = chi)
            chi = int(round(math.exp(rng.uniform(math.log(4), math.log(20)))))
            n = chi * chi if rng.random() < 0.6 else chi
            return {"kind": kind, "prec": "f64", "chi_b": chi, "n": n, "kappa": float(10 ** rng.uniform(0.5, 4.0))}
        prec = rng.choice(["f64", "f64", "f64", "bf16x3", "bf16x3", "oz4", "tf32", "bf16", "oz3", "bf16x6"])
        top = {"sweep": 12, "energy_grad": 16}.get(kind, 16 if prec == "f64" else 32)
        chi = int(round(math.exp(rng.uniform(math.log(4), math.log(top)))))
        if kind == "sweep":
            case = {"kind": kind, "prec": prec, "chi_t": chi, "graph": rng.random() < 0.5}
        elif kind == "fixed_point":
            case = {"kind": kind, "prec": prec, "chi_b": chi, "chi_t": chi}
        else:  # some transitional layers, whose upper legs are wider than the lower ones
            chi_b = chi if rng.random() < 0.7 else max(4, int(round(chi * rng.uniform(0.4, 1.0))))
            case = {"kind": kind, "prec": prec, "chi_b": chi_b, "chi_t": min(chi, chi_b * chi_b)}
        if _seconds(case) <= cap:
            return case


# ---------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------
def _dims(case):
    return M.layer_dims(case["chi_t"], N_LAYERS)


def _isometry(gen, rows, cols):
    q, _ = torch.linalg.qr(torch.randn(rows, cols, dtype=torch.float64, device="cuda", generator=gen))
    return q[:, :cols].contiguous()


def _operator(gen, chi):
    """A symmetric 3-site operator, shifted to be mostly negative as the library's Hamiltonian densities are."""
    n = chi ** 3
    x = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=gen)
    x = (x + x.T).div_(math.sqrt(8.0 * n))
    x.diagonal().sub_(1.0)
    return x.reshape(-1)


def _density(gen, chi):
    """A 3-site density matrix with a decaying spectrum over a full-rank floor, unit trace."""
    n = chi ** 3
    r = min(n, 64)
    v = torch.randn(n, r, dtype=torch.float64, device="cuda", generator=gen)
    v *= torch.exp(-0.1 * torch.arange(r, dtype=torch.float64, device="cuda"))
    x = v @ v.T
    x.diagonal().add_(1e-3)
    x /= x.diagonal().sum()
    return x.reshape(-1)


def _inputs(case, seed):
    """h, rho, u, w of one layer."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    cb, ct = case["chi_b"], case["chi_t"]
    s = {"u": _isometry(gen, cb * cb, cb * cb).reshape(-1), "w": _isometry(gen, cb * cb, ct).reshape(-1)}
    kind = case["kind"]
    if kind in ("ascend", "noalloc", "env_u", "env_w", "energy_grad"):
        s["h"] = _operator(gen, cb)
    if kind in ("descend", "env_u", "env_w", "energy_grad"):
        s["rho"] = _density(gen, ct)
    return s


def _environment(case, seed):
    """An m x n environment whose singular values decay geometrically over the factor kappa."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    m, n = case["chi_b"] ** 2, case["n"]
    s = case["kappa"] ** (-torch.arange(n, dtype=torch.float64, device="cuda") / max(1, n - 1))
    return ((_isometry(gen, m, n) * s) @ _isometry(gen, n, n).T).contiguous()


def _hamiltonian():
    h1, shift = G.mera_ising_h1(1.0)
    return torch.from_numpy(np.ascontiguousarray(h1)).reshape(-1), shift


def _mera(case, seed):
    """Seeded tensors of every layer (numpy), as an optimisation starts from."""
    return M.init_mera(seed, case["chi_t"], N_LAYERS)


def prepare(case, seed):
    kind, prec = case["kind"], G.PRECS[case["prec"]]
    new = lambda *n: torch.empty(*n, dtype=torch.float64, device="cuda")  # noqa: E731
    if kind == "polar":
        m, n = case["chi_b"] ** 2, case["n"]
        return {"case": case, "env": _environment(case, seed).reshape(-1), "m": m, "n": n, "out": new(m * n),
                "ws": G.workspace(G.mera_polar_workspace_size(m, n))}
    if kind == "sweep":
        chi = case["chi_t"]
        layers = _mera(case, seed)
        dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
        us, ws = [dev(u) for u, _ in layers], [dev(w) for _, w in layers]
        rho = (torch.eye(chi ** 3, dtype=torch.float64, device="cuda") / chi ** 3).contiguous()
        st = G.MeraState(us, ws, rho)
        h1, shift = _hamiltonian()
        s = {"case": case, "prec": prec, "mera": st, "h1": h1.cuda(), "shift": shift, "e": new(1),
             "ws": G.workspace(G.mera_sweep_workspace_size(st.chi_b, st.chi_t, prec))}
        if case["graph"]:
            stream = torch.cuda.Stream()
            torch.cuda.synchronize()
            s["graph"] = G.mera_sweep_graph(st, s["h1"], shift, N_POW, s["e"], prec=prec, ws=s["ws"], stream=stream)
        return s
    cb, ct = case["chi_b"], case["chi_t"]
    s = {"case": case, "prec": prec, **_inputs(case, seed)}
    if kind == "noalloc":
        s["out"] = new(ct ** 6)
    elif kind == "energy_grad":
        for k in ("h", "rho", "u", "w"):
            s[k].requires_grad_(True)
    elif kind == "fixed_point":
        n = ct ** 3
        s["start"] = (torch.eye(n, dtype=torch.float64, device="cuda") / n).reshape(-1)
        s["rho"] = s["start"].clone()
        s["ws"] = G.workspace(G.mera_workspace_size(G.OP_FIXED_POINT, cb, ct, prec))
    else:
        s["out"] = new({"ascend": ct ** 6, "descend": cb ** 6, "env_u": cb ** 4, "env_w": cb ** 2 * ct}[kind])
        s["ws"] = G.workspace(G.mera_workspace_size(MAPS[kind], cb, ct, prec))
    return s


# ---------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "polar":
        return G.mera_polar_update(s["env"], s["m"], s["n"], s["out"], ws=s["ws"])
    if kind == "sweep":
        st = s["mera"]
        if case["graph"]:
            s["graph"].launch()
        else:
            G.mera_sweep(st, s["h1"], s["shift"], N_POW, s["e"], prec=s["prec"], ws=s["ws"])
        return {"energy": s["e"], "u": st.us, "w": st.ws, "rho_star": st.rho_star}
    cb, ct, prec = case["chi_b"], case["chi_t"], s["prec"]
    if kind == "noalloc":
        return G.mera_ascend_noalloc(s["h"], s["u"], s["w"], cb, ct, s["out"], prec=prec)
    if kind == "ascend":
        return G.mera_ascend(s["h"], s["u"], s["w"], cb, ct, s["out"], prec=prec, ws=s["ws"])
    if kind == "descend":
        return G.mera_descend(s["rho"], s["u"], s["w"], cb, ct, s["out"], prec=prec, ws=s["ws"])
    if kind == "env_u":
        return G.mera_env_u(s["h"], s["rho"], s["u"], s["w"], cb, ct, s["out"], prec=prec, ws=s["ws"])
    if kind == "env_w":
        return G.mera_env_w(s["h"], s["rho"], s["u"], s["w"], cb, ct, s["out"], prec=prec, ws=s["ws"])
    if kind == "fixed_point":  # from the maximally mixed state, as an optimisation's first sweep does
        s["rho"].copy_(s["start"])
        return G.mera_fixed_point_rho(s["u"], s["w"], ct, s["rho"], N_POW, prec=prec, ws=s["ws"])
    x = [s[k] for k in ("h", "rho", "u", "w")]  # energy_grad
    e = A.mera_energy(*x, cb, ct, prec)
    return [e.detach()] + list(torch.autograd.grad(e, x))


# ---------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "polar":  # read and write the matrix; flops of a singular value decomposition and U V^T
        m, n = case["chi_b"] ** 2, case["n"]
        return {"bytes": 16.0 * m * n, "flops": 8.0 * m * n * n + 20.0 * n ** 3}
    if kind == "sweep":
        flops = size = 0.0
        for k, (cb, ct) in enumerate(_dims(case)):
            f = {name: G.mera_flops(op, cb, ct) for name, op in MAPS.items()}
            flops += f["env_u"] + f["env_w"]
            flops += 2 * f["ascend"] if k + 1 < N_LAYERS else N_POW * f["descend"]
            size += 16.0 * (cb ** 4 + cb ** 2 * ct)  # u and w, read and written
        return {"bytes": size + 16.0 * case["chi_t"] ** 6 + 8.0 * 4 ** 6, "flops": flops}
    cb, ct = case["chi_b"], case["chi_t"]
    tensors, h, rho = cb ** 4 + cb ** 2 * ct, cb ** 6, ct ** 6
    f = {name: G.mera_flops(op, cb, ct) for name, op in MAPS.items()}
    if kind in ("ascend", "noalloc", "descend"):
        return {"bytes": 8.0 * (tensors + h + rho), "flops": f["descend" if kind == "descend" else "ascend"]}
    if kind == "env_u":
        return {"bytes": 8.0 * (tensors + h + rho + cb ** 4), "flops": f["env_u"]}
    if kind == "env_w":
        return {"bytes": 8.0 * (tensors + h + rho + cb ** 2 * ct), "flops": f["env_w"]}
    if kind == "fixed_point":
        return {"bytes": 8.0 * (tensors + 2 * rho), "flops": N_POW * f["descend"]}
    # energy_grad: symmetric or not, the entry point serves both, so both halves of each environment are needed
    return {"bytes": 16.0 * (tensors + h + rho),
            "flops": 2 * f["ascend"] + f["descend"] + 2 * f["env_u"] + 2 * f["env_w"]}


# ---------------------------------------------------------------------------------------------------------------
# the same in 64 bits, with plain torch
# ---------------------------------------------------------------------------------------------------------------
# Networks of the even and the odd position (Sec. II B and Fig. 4 of the paper): ket isometries and disentanglers,
# the operator, bra disentanglers and isometries; the density closes the energy.
KET_W, BRA_W = ("xap", "bcq", "dyr"), ("xAs", "BCt", "Dyv")
KET_U, BRA_U = (("eiab", "jkcd"), ("ijab", "kecd")), (("elAB", "mnCD"), ("lmAB", "neCD"))


def _order(legs, out, dim):
    """Pairwise contraction order of the least flops, by dynamic programming over subsets of the tensors."""
    n, full = len(legs), (1 << len(legs)) - 1
    sets = [frozenset(x) for x in legs]
    opens = [frozenset()] * (full + 1)
    for s in range(1, full + 1):
        opens[s] = opens[s & (s - 1)] ^ sets[(s & -s).bit_length() - 1]
    opens[full] = frozenset(out)
    size = {}

    def volume(k):
        if k not in size:
            size[k] = math.prod(dim[c] for c in k)
        return size[k]

    best = {1 << k: (0.0, None) for k in range(n)}
    for s in sorted(range(1, full + 1), key=lambda v: bin(v).count("1")):
        if s in best or (len(opens[s]) > 7 and s != full):
            continue
        t = (s - 1) & s
        while t:
            o = s ^ t
            if t > o and t in best and o in best and opens[t] & opens[o]:
                c = best[t][0] + best[o][0] + volume(opens[t] | opens[o])
                if s not in best or c < best[s][0]:
                    best[s] = (c, t)
            t = (t - 1) & s
    return best, opens, full


def _contract(tensors, legs, out, dim):
    best, opens, full = _order(legs, out, dim)

    def value(s):
        if best[s][1] is None:
            k = s.bit_length() - 1
            return tensors[k], legs[k]
        (x, a), (y, b) = value(best[s][1]), value(s ^ best[s][1])
        k = [c for c in a if c in b]
        ra, rb = [c for c in a if c not in k], [c for c in b if c not in k]
        kk = math.prod(dim[c] for c in k)
        x = x.permute([a.index(c) for c in ra + k]).reshape(-1, kk)
        y = y.permute([b.index(c) for c in k + rb]).reshape(kk, -1)
        return (x @ y).reshape([dim[c] for c in ra + rb]), "".join(ra + rb)

    x, a = value(full)
    return x.permute([a.index(c) for c in out])


def _map(kind, h, rho, u, w, cb, ct):
    """The mean over the two positions of a superoperator, or the summed environment."""
    dim = {c: (ct if c in "pqrstv" else cb) for c in "abcdeijklmnpqrstvxyABCD"}
    h = None if h is None else h.reshape((cb,) * 6)
    rho = None if rho is None else rho.reshape((ct,) * 6)
    u, w = u.reshape((cb,) * 4), w.reshape(cb, cb, ct)
    total = 0.0
    for p in (0, 1):
        for hole in range({"env_u": 2, "env_w": 3}.get(kind, 1)):
            net = [(w, x) for x in KET_W] + [(u, x) for x in KET_U[p]]
            if kind != "descend":
                net.append((h, "ijklmn"))
            net += [(u, x) for k, x in enumerate(BRA_U[p]) if not (kind == "env_u" and k == hole)]
            net += [(w, x) for k, x in enumerate(BRA_W) if not (kind == "env_w" and k == hole)]
            if kind == "descend":
                net.append((rho, "pqrstv"))
            elif kind != "ascend":
                net.append((rho, "stvpqr"))
            out = {"ascend": "pqrstv", "descend": "ijklmn", "env_u": BRA_U[p][hole % 2], "env_w": BRA_W[hole]}[kind]
            total = total + 0.5 * _contract([x for x, _ in net], [x for _, x in net], out, dim)
    return total.reshape(-1)


def _fixed_point(rho, u, w, chi):
    n = chi ** 3
    for _ in range(N_POW):
        x = _map("descend", None, rho, u, w, chi, chi).reshape(n, n)
        rho = (x + x.T) / (2.0 * x.diagonal().sum())
    return rho.reshape(-1)


def _polar(env, m, n):
    # the decomposition runs on the host, where it is the reference one
    a, _, b = torch.linalg.svd(env.reshape(m, n).cpu(), full_matrices=False)
    return -(a @ b).cuda()


def _energy(h, rho, u, w, cb, ct):
    n = ct ** 3
    return (_map("ascend", h, None, u, w, cb, ct).reshape(n, n) * rho.reshape(n, n).T).sum()


def _sweep(case, seed):
    layers, dims = _mera(case, seed), _dims(case)
    us = [torch.from_numpy(np.ascontiguousarray(u)).cuda() for u, _ in layers]
    ws = [torch.from_numpy(np.ascontiguousarray(w)).cuda() for _, w in layers]
    h1, shift = _hamiltonian()
    hs = [h1.cuda()]
    for t in range(N_LAYERS - 1):
        hs.append(_map("ascend", hs[t], None, us[t], ws[t], *dims[t]))
    chi = case["chi_t"]
    star = _fixed_point(torch.eye(chi ** 3, dtype=torch.float64, device="cuda") / chi ** 3, us[-1], ws[-1], chi)
    rho = star
    for t in reversed(range(N_LAYERS)):
        cb, ct = dims[t]
        us[t] = _polar(_map("env_u", hs[t], rho, us[t], ws[t], cb, ct), cb * cb, cb * cb).reshape(us[t].shape)
        ws[t] = _polar(_map("env_w", hs[t], rho, us[t], ws[t], cb, ct), cb * cb, ct).reshape(ws[t].shape)
        if 0 < t < N_LAYERS - 1:
            rho = _map("descend", None, rho, us[t], ws[t], cb, ct)
    e = 0.5 * (_energy(hs[0], rho, us[0], ws[0], *dims[0]) + shift)
    return {"energy": e.reshape(1), "u": us, "w": ws, "rho_star": star.reshape(-1)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "polar":
        m, n = case["chi_b"] ** 2, case["n"]
        return _polar(_environment(case, seed), m, n).reshape(-1)
    if work(case)["flops"] > 1.3e13:  # over about twelve seconds in 64 bits
        return None
    if kind == "sweep":
        return _sweep(case, seed)
    cb, ct = case["chi_b"], case["chi_t"]
    s = _inputs(case, seed)
    h, rho, u, w = s.get("h"), s.get("rho"), s["u"], s["w"]
    if kind == "fixed_point":
        n = ct ** 3
        return _fixed_point(torch.eye(n, dtype=torch.float64, device="cuda") / n, u, w, ct)
    if kind != "energy_grad":
        return _map("ascend" if kind == "noalloc" else kind, h, rho, u, w, cb, ct)
    ht, rt = h.reshape(cb ** 3, -1).T.contiguous().reshape(-1), rho.reshape(ct ** 3, -1).T.contiguous().reshape(-1)
    return [_energy(h, rho, u, w, cb, ct), _map("descend", None, rt, u, w, cb, ct), _map("ascend", ht, None, u, w, cb, ct),
            _map("env_u", h, rho, u, w, cb, ct) + _map("env_u", ht, rt, u, w, cb, ct),
            _map("env_w", h, rho, u, w, cb, ct) + _map("env_w", ht, rt, u, w, cb, ct)]
