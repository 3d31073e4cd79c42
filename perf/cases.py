"""The calls that a user of the trace estimator makes, as cases whose time can be measured.

A case is a dict of plain values; ``prepare`` makes what a program holds before the call (the
hierarchy, device vectors, network weights), ``run`` makes the call through the ctypes binding
and returns what it computes, ``work`` gives the bytes and operations of one pass that no
implementation can do without, and ``exact`` the values in 64 bits where plain numpy / torch
can give them in seconds.

Kinds of calls:
  estimate  one whole trace estimate (Secs. 2 and 5)
  samples   one block of level-difference samples with its statistics (Remark 4.3)
  solve     one batched level solve (Remark 4.1)
  apply     one level operator applied to a block of vectors (Examples 5.1 and 5.3)
  dense     the coarsest level's dense product Y = A B in single precision
  net, grad the learned correction: its forward pass, and its loss gradient (a training step)
  setup     the construction of a hierarchy (Sec. 4.1)
"""
import math

import numpy as np
import torch

from paper_2108_11281_gb300 import mlmc
from paper_2108_11281_gb300.workloads import LAPLACE_1024, WILSON_128, WILSON_256, gauge_links

AGG = 4          # aggregates of 4 x 4 sites on every level
N_TV = 4         # test vectors per aggregate


def listed():
    return [
        # the headline: tr(A^-1) of the 1024^2 Laplacian to 1e-3 with the optimal allocation; samples1..3
        # are the counts that this allocation reaches (they size work(); the call decides for itself)
        dict(name="estimate_laplace_1024", kind="estimate", op="laplace", side=LAPLACE_1024["nx"], levels=4,
             mixed=True, block=64, coarse_block=128, growth=2, fixed=False, samples1=64, samples2=128, samples3=1024),
        # the Wilson / Schwinger operator with Z4 noise on a fixed sample budget
        dict(name="estimate_wilson_128", kind="estimate", op="wilson", side=WILSON_128["nx"], levels=3, mixed=True,
             block=32, coarse_block=128, growth=0, fixed=True, samples1=128, samples2=512, samples3=0, tuned=True),
        # the paper's own bilinear hierarchy: one block of hat-form samples on the second difference,
        # odd grid sides, as a sharded or resumed estimate draws them
        dict(name="samples_bilinear_511", kind="samples", op="bilinear", side=511, levels=6, mixed=True, level=2, k=48),
        # the smallest calls: a block on a 64^2 Laplacian with piecewise-constant P in double precision
        dict(name="samples_laplace_64", kind="samples", op="constant", side=64, levels=2, mixed=False, level=1, k=64),
        # a program's own right-hand sides, double precision throughout, ragged block
        dict(name="solve_laplace_192_f64", kind="solve", op="laplace", side=192, levels=3, mixed=False, k=21),
        # a program's own right-hand sides for the Wilson operator, mixed precision
        dict(name="solve_wilson_64", kind="solve", op="wilson", side=64, levels=3, mixed=True, k=32),
        # operator products in double precision: the largest fine level, and a coarse level of 8 x 8 blocks
        dict(name="apply_laplace_1024", kind="apply", op="constant", side=1024, levels=4, level=1, k=64),
        dict(name="apply_wilson_coarse", kind="apply", op="wilson", side=128, levels=3, level=2, k=128),
        # the coarsest solve of a cycle, at the size the 1024^2 hierarchy has
        dict(name="dense_1024", kind="dense", complex=False, n=1024, k=128),
        # the learned correction on the 256^2 Wilson lattice: inference and one training gradient
        dict(name="net_wilson_256", kind="net", side=WILSON_256["nx"], k=WILSON_256["block"]),
        dict(name="grad_wilson_128", kind="grad", side=128, k=32),
        # building the hierarchy of the headline estimate, which every new operator pays once
        dict(name="setup_laplace_1024", kind="setup", op="laplace", side=1024, levels=4, mixed=True, block=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same calls over the lattice sides, levels, block widths, sample budgets and
    precisions in use (sides are the multiples that the coarsening needs; widths and budgets are any)."""
    kind = rng.choice(["estimate", "samples", "solve", "apply", "dense", "net", "grad", "setup"])
    if kind == "estimate":
        if rng.random() < 0.5:
            levels = rng.choice([3, 4])
            side = 64 * rng.randint(3, 14) if levels == 4 else 16 * rng.randint(4, 16)
            return dict(kind=kind, op="laplace", side=side, levels=levels, mixed=rng.random() < 0.75,
                        block=rng.choice([16, 32, 64]), coarse_block=rng.choice([64, 128]), growth=rng.randint(0, 1),
                        fixed=True, samples1=rng.randint(16, 64), samples2=rng.randint(16, 128),
                        samples3=rng.randint(16, 128) if levels == 4 else 0)
        return dict(kind=kind, op="wilson", side=16 * rng.randint(3, 8), levels=3, mixed=True,
                    block=rng.choice([16, 32]), coarse_block=rng.choice([32, 64, 128]), growth=0, fixed=True,
                    samples1=rng.randint(16, 64), samples2=rng.randint(16, 128), samples3=0)
    if kind == "samples":
        if rng.random() < 0.5:
            levels = rng.randint(3, 6)
            side = 2 ** (levels - 1) * (rng.randint(7, 15) + 1) - 1
            return dict(kind=kind, op="bilinear", side=side, levels=levels, mixed=rng.random() < 0.75,
                        level=rng.randint(1, levels - 1), k=_log_int(rng, 4, 64))
        return dict(kind=kind, op="constant", side=8 * rng.randint(3, 16), levels=2, mixed=rng.random() < 0.5, level=1,
                    k=_log_int(rng, 4, 64))
    if kind == "solve":
        op = rng.choice(["laplace", "wilson"])
        side = 16 * (_log_int(rng, 4, 16) if op == "laplace" else rng.randint(2, 4))
        return dict(kind=kind, op=op, side=side, levels=3, mixed=rng.random() < 0.6, k=_log_int(rng, 1, 64))
    if kind == "apply":
        if rng.random() < 0.5:
            return dict(kind=kind, op="constant", side=64 * _log_int(rng, 1, 16), levels=4, level=1,
                        k=_log_int(rng, 1, 64))
        return dict(kind=kind, op=rng.choice(["laplace", "wilson"]), side=16 * _log_int(rng, 3, 8), levels=3,
                    level=rng.randint(1, 2), k=_log_int(rng, 1, 128))
    if kind == "dense":
        cplx = rng.random() < 0.5
        return dict(kind=kind, complex=cplx, n=_log_int(rng, 64, 1024 if cplx else 2048), k=_log_int(rng, 1, 256))
    if kind in ("net", "grad"):
        return dict(kind=kind, side=16 * _log_int(rng, 2, 12), k=_log_int(rng, 4, 32))
    return dict(kind="setup", op=rng.choice(["laplace", "wilson"]), side=16 * _log_int(rng, 3, 8), levels=3,
                mixed=rng.random() < 0.75, block=rng.choice([16, 32, 64]))


# ------------------------------------------------------------------ what a program holds before the call
def _params(c, **kw):
    """Hierarchy parameters of the case's operator class: the settings the estimates use."""
    p = dict(levels=c["levels"], agg_x=AGG, agg_y=AGG, kcycle_its=2, max_iter=5000, fgmres_restart=8, inner_its=8,
             smooth_pre=2, smooth_post=2,
             precision=mlmc.PREC_MIXED_FP32 if c.get("mixed", True) else mlmc.PREC_FP64)
    if c["op"] == "laplace":
        p.update(n_tv=N_TV, setup_kind=mlmc.SETUP_SMOOTH, setup_sweeps=160, coarse_sweeps=20, bootstrap=2, boot_iters=5,
                 reorth=0)
    elif c["op"] == "wilson":
        p.update(n_tv=N_TV, spin_split=1, setup_kind=mlmc.SETUP_INVERSE, setup_sweeps=20, coarse_sweeps=10,
                 setup_omega=1.0, bootstrap=4, boot_iters=4, fgmres_restart=10)
    elif c["op"] == "constant":
        p.update(n_tv=1, setup_kind=mlmc.SETUP_CONSTANT, bootstrap=0, smooth_pre=1, smooth_post=1)
    else:
        p.update(n_tv=1, transfer=mlmc.TRANSFER_BILINEAR, bootstrap=0, smooth_pre=1, smooth_post=1)
    p.update(kw)
    return mlmc.default_params(**p)


def _wilson_links(side):
    return gauge_links(side, side, WILSON_128["link_sd"], WILSON_128["link_seed"])


def _mass(c):
    """The mass tuned to a condition of 1e3 on the 128^2 configuration; a more regular one elsewhere."""
    return WILSON_128["mass"] if c.get("tuned") else -0.10


def _hierarchy(c, **kw):
    if c["op"] == "wilson":
        return mlmc.Hierarchy(mlmc.OP_WILSON2D, c["side"], c["side"], _params(c, **kw), mass=_mass(c),
                              links=_wilson_links(c["side"]))
    return mlmc.Hierarchy(mlmc.OP_LAPLACE2D, c["side"], c["side"], _params(c, **kw))


def _randn(shape, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn(*shape, dtype=dtype, device="cuda", generator=g)


def _net_weights(seed):
    """Weights of the c0 -> 16 -> 16 -> c0 network (c0 = 4: two complex spins), [c_out][c_in][3][3] each."""
    rng = np.random.default_rng([int(seed), 3])
    return [(rng.standard_normal((co, ci, 3, 3)) * math.sqrt(1.0 / (9 * ci))).astype(np.float32)
            for co, ci in ((16, 4), (16, 16), (4, 16))]


def _dense_inputs(c, seed):
    dt = torch.complex64 if c["complex"] else torch.float32
    return _randn((c["n"], c["n"]), dt, seed) / math.sqrt(c["n"]), _randn((c["n"], c["k"]), dt, seed + 1)


def _rhs(c, seed):
    n = c["side"] ** 2 * (2 if c["op"] == "wilson" else 1)
    return _randn((n, c["k"]), torch.complex128 if c["op"] == "wilson" else torch.float64, seed)


def _residuals(c, seed):
    return _randn((2 * c["side"] ** 2, c["k"]), torch.complex64, seed)


def prepare(c, seed):
    kind, s = c["kind"], {"case": c, "seed": int(seed)}
    if kind == "estimate":
        s["h"] = _hierarchy(c, block=c["block"], coarse_block=c["coarse_block"], coarse_growth=c["growth"])
    elif kind == "samples":
        s["h"] = _hierarchy(c, block=c["k"])
    elif kind == "solve":
        s["h"], s["b"] = _hierarchy(c, block=c["k"]), _rhs(c, seed)
        s["x"] = torch.empty_like(s["b"])
    elif kind == "apply":
        # products alone: narrow blocks for the solver's own buffers, and no test-vector refinement
        s["h"] = _hierarchy(c, block=8, bootstrap=0)
        s["x"] = _randn((s["h"].n(c["level"]), c["k"]), torch.complex128 if c["op"] == "wilson" else torch.float64, seed)
        s["y"] = torch.empty_like(s["x"])
    elif kind == "dense":
        s["A"], s["B"] = _dense_inputs(c, seed)
        s["Y"] = torch.empty_like(s["B"])
    elif kind in ("net", "grad"):
        s["h"] = _hierarchy(dict(op="wilson", kind=kind, levels=3, side=c["side"]), block=c["k"], bootstrap=0)
        s["h"].learned_set(np.concatenate([w.ravel() for w in _net_weights(seed)]), enable=1)
        s["r"] = _residuals(c, seed)
        s["e"] = torch.empty_like(s["r"])
    else:
        s["seed"] = int(seed) % (1 << 31)      # the random test vectors' stream
    torch.cuda.synchronize()
    return s


def run(s):
    c, kind, h = s["case"], s["case"]["kind"], s.get("h")
    if kind == "estimate":
        budget = [c["samples%d" % i] for i in range(1, c["levels"])]
        kw = dict(allocation=mlmc.ALLOC_FIXED, n_fixed=budget) if c["fixed"] else \
            dict(allocation=mlmc.ALLOC_OPTIMAL, cost_model=mlmc.COST_NOMINAL, eps=LAPLACE_1024["eps"])
        r = mlmc.result_dict(h.trace_estimate(noise=mlmc.NOISE_Z4 if c["op"] == "wilson" else mlmc.NOISE_RADEMACHER,
                                              seed=s["seed"], tol=LAPLACE_1024["tol"], **kw))
        return {"trace": np.array([r["trace"]]), "std_err": np.array([r["std_err"]]), "mean": np.array(r["mean"]),
                "variance": np.array(r["variance"]), "n_samples": np.array(r["n_samples"])}
    if kind == "samples":
        form = mlmc.FORM_HAT if c["op"] == "bilinear" else mlmc.FORM_SIMPLIFIED
        x, (count, mean, m2), _ = h.sample_block(c["level"], form, mlmc.NOISE_RADEMACHER, s["seed"], 0, c["k"], 1e-11)
        return {"samples": x, "mean": np.array([mean]), "m2": np.array([m2]), "count": int(count)}
    if kind == "solve":
        h.solve(1, s["b"].data_ptr(), s["x"].data_ptr(), c["k"], 1e-11)
        return s["x"]
    if kind == "apply":
        h.apply(c["level"], s["x"].data_ptr(), s["y"].data_ptr(), c["k"])
        return s["y"]
    if kind == "dense":
        mlmc.dense_apply(c["complex"], s["A"].data_ptr(), s["B"].data_ptr(), s["Y"].data_ptr(), c["n"], c["k"])
        return s["Y"]
    if kind == "net":
        h.learned_apply(s["r"].data_ptr(), s["e"].data_ptr(), c["k"])
        return s["e"]
    if kind == "grad":
        loss, g = h.learned_grad(s["r"].data_ptr(), c["k"])
        return {"loss": loss, "grad": g}
    h = _hierarchy(c, block=c["block"], setup_seed=s["seed"])
    out = {"coarse_trace": np.array([h.coarse_trace_exact()]), "coarse_operator": h.operator(c["levels"])}
    h.close()
    return out


# ------------------------------------------------------------------ what one pass cannot do without
def _level_sizes(c):
    """(unknowns, matrix entries per row) of each level."""
    out, side = [], c["side"]
    for l in range(c["levels"]):
        if c["op"] == "bilinear":
            out.append((side * side, 5 if l == 0 else 9))
            side = (side - 1) // 2
        else:
            dc = {"laplace": N_TV, "wilson": 2 * N_TV, "constant": 1}[c["op"]]
            d = {"wilson": 2}.get(c["op"], 1) if l == 0 else dc
            out.append((side * side * d, 9 if l == 0 and c["op"] == "wilson" else 5 * d))
            side //= AGG
    return out


def work(c):
    """A sample: its noise block and its solution, written and read once on both levels, and one product with
    each operator; a solve: its right-hand sides read, its solution written, one product (the residual)."""
    kind = c["kind"]
    if kind == "dense":
        z, m = (8, 8) if c["complex"] else (4, 2)
        return {"bytes": z * (c["n"] ** 2 + 2 * c["n"] * c["k"]), "flops": m * c["n"] ** 2 * c["k"]}
    if kind in ("net", "grad"):
        pairs, macs = c["side"] ** 2 * c["k"], 9 * (4 * 16 + 16 * 16 + 16 * 4)
        if kind == "net":
            return {"bytes": 2 * 16 * pairs, "flops": 2 * macs * pairs}
        # forward, the weight gradients of all layers, the data gradients of the last two
        return {"bytes": 16 * pairs, "flops": 2 * (3 * macs - 9 * 4 * 16) * pairs}
    lv, cplx = _level_sizes(c), c["op"] == "wilson"
    z, m = (16, 8) if cplx else (8, 2)
    if kind == "apply":
        n, row = lv[c["level"] - 1]
        matrix = 0 if c["op"] != "wilson" and c["level"] == 1 else n * row * z
        return {"bytes": 2 * n * c["k"] * z + matrix, "flops": m * n * row * c["k"]}
    if kind == "solve":
        n, row = lv[0]
        return {"bytes": 2 * n * c["k"] * z, "flops": m * n * row * c["k"]}
    if kind == "setup":
        # the test vectors filtered once, every level's operator written, the coarsest inverse
        n, nl = lv[0][0], lv[-1][0]
        return {"bytes": z * (2 * N_TV * n + sum(a * r for a, r in lv) + 2 * nl * nl), "flops": m * nl ** 3}
    counts = [c["samples%d" % i] for i in range(1, c["levels"])] if kind == "estimate" else \
        [c["k"] if l == c["level"] else 0 for l in range(1, c["levels"])]
    by = sum(N * 4 * z * (lv[l][0] + lv[l + 1][0]) for l, N in enumerate(counts))
    fl = sum(N * m * (lv[l][0] * lv[l][1] + lv[l + 1][0] * lv[l + 1][1]) for l, N in enumerate(counts))
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ the values in 64 bits
def _second_difference(n):
    return 2.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1)


def _kron_pair(T, M):
    """(V, w) with (T x M + M x T)^-1 = (V x V) diag(1 / (w_i + w_j)) (V x V)^T, by T v = w M v."""
    L = np.linalg.cholesky(M)
    w, Q = np.linalg.eigh(np.linalg.solve(L, np.linalg.solve(L, T).T))
    return np.linalg.solve(L.T, Q), w


def _quadratic(x, V, w):
    """x^T A^-1 x for each x (count, n, n) and A as in _kron_pair."""
    c = np.einsum("ai,sab,bj->sij", V, x, V, optimize=True)
    return (c * c / (w[:, None] + w[None, :])).sum(axis=(1, 2))


def _mulhilo(a, b):
    """High and low 64 bits of a * b."""
    m = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    al, ah, bl, bh = a & m, a >> s, b & m, b >> s
    mid = ah * bl + ((al * bl) >> s)
    mid2 = al * bh + (mid & m)
    return ah * bh + (mid >> s) + (mid2 >> s), a * b


def _rademacher(n, seed, level, k):
    """Samples 0..k-1 of the Philox4x64-10 sign stream: bit b of word q of counter (block, sample) is row
    256 block + 64 q + b, key (seed, level)."""
    blocks = (n + 255) // 256
    with np.errstate(over="ignore"):
        c = [np.broadcast_to(np.arange(blocks, dtype=np.uint64), (k, blocks)).copy(),
             np.broadcast_to(np.arange(k, dtype=np.uint64)[:, None], (k, blocks)).copy(),
             np.zeros((k, blocks), np.uint64), np.zeros((k, blocks), np.uint64)]
        key = [np.uint64(seed), np.uint64(level)]
        for r in range(10):
            if r:
                key = [key[0] + np.uint64(0x9E3779B97F4A7C15), key[1] + np.uint64(0xBB67AE8584CAA73B)]
            h0, l0 = _mulhilo(np.uint64(0xD2E7470EE14C6C93), c[0])
            h1, l1 = _mulhilo(np.uint64(0xCA5A826395121157), c[2])
            c = [h1 ^ c[1] ^ key[0], l1, h0 ^ c[3] ^ key[1], l0]
    words = np.stack(c, axis=-1)
    bits = (words[..., None] >> np.arange(64, dtype=np.uint64)) & np.uint64(1)
    return 1.0 - 2.0 * bits.reshape(k, blocks * 256)[:, :n].astype(np.float64)


def _samples_exact(c, seed):
    n = c["side"]
    x = _rademacher(n * n, seed, c["level"], c["k"]).reshape(c["k"], n, n)
    T, M = _second_difference(n), np.eye(n)
    pair = []
    for l in range(1, c["level"] + 2):
        if l >= c["level"]:
            V, w = _kron_pair(T, M)
            pair.append(_quadratic(x, V, w))
        if c["op"] == "bilinear":
            p = np.zeros((n, (n - 1) // 2))
            for i in range(p.shape[1]):
                p[2 * i:2 * i + 3, i] = 0.5, 1.0, 0.5
        else:
            p = np.kron(np.eye(n // AGG), np.full((AGG, 1), 0.5))
        x, T, M, n = np.einsum("ai,sab,bj->sij", p, x, p, optimize=True), p.T @ T @ p, p.T @ M @ p, p.shape[1]
    s = pair[0] - pair[1]
    return {"samples": s.astype(np.complex128), "mean": np.array([s.mean() + 0j]),
            "m2": np.array([((s - s.mean()) ** 2).sum()]), "count": None}


def _wilson(u, U, mass):
    """The Wilson operator of Example 5.3 on u (ny, nx, 2, k), links U (2, ny, nx)."""
    s1 = torch.tensor([[0, 1], [1, 0]], dtype=u.dtype, device=u.device)
    s2 = torch.tensor([[0, 1j], [-1j, 0]], dtype=u.dtype, device=u.device)
    one = torch.eye(2, dtype=u.dtype, device=u.device)
    out = (4.0 + mass) * u
    for axis, link, s in ((1, U[0], s1), (0, U[1], s2)):
        hop = link[:, :, None, None] * torch.einsum("ab,yxbk->yxak", one - s, torch.roll(u, -1, axis))
        back = torch.roll(link.conj()[:, :, None, None] * torch.einsum("ab,yxbk->yxak", one + s, u), 1, axis)
        out = out - hop - back
    return out


def _laplace(u):
    """The Dirichlet Laplacian of Example 5.1 on u (ny, nx, k)."""
    p = torch.nn.functional.pad(u, (0, 0, 1, 1, 1, 1))
    return 4.0 * u - p[1:-1, 2:] - p[1:-1, :-2] - p[2:, 1:-1] - p[:-2, 1:-1]


def _net(r, Ws, side):
    """Three 3 x 3 periodic convolutions with a ReLU after the first two on r (sites * 2, k) complex."""
    a = torch.view_as_real(r).reshape(side, side, 2, -1, 2).permute(3, 2, 4, 0, 1).reshape(-1, 4, side, side)
    for i, W in enumerate(Ws):
        a = torch.nn.functional.conv2d(torch.nn.functional.pad(a, (1, 1, 1, 1), mode="circular"), W)
        a = torch.relu(a) if i < 2 else a
    a = a.reshape(-1, 2, 2, side, side).permute(3, 4, 1, 0, 2).contiguous()
    return torch.view_as_complex(a).reshape(side * side * 2, -1)


def exact(c, seed):
    kind, side = c["kind"], c.get("side")
    if kind == "samples":
        return _samples_exact(c, seed)
    if kind == "dense":
        A, B = _dense_inputs(c, seed)
        wide = torch.complex128 if c["complex"] else torch.float64
        return A.to(wide) @ B.to(wide)
    if kind in ("net", "grad"):
        r = _residuals(c, seed).to(torch.complex128)
        Ws = [torch.tensor(w, dtype=torch.float64, device="cuda", requires_grad=kind == "grad") for w in _net_weights(seed)]
        parts = [(_net(q, Ws, side), q) for q in r.split(8, dim=1)] if kind == "net" else []
        if kind == "net":
            return torch.cat([e for e, _ in parts], dim=1)
        U = torch.tensor(_wilson_links(side), device="cuda")
        loss = 0.0
        for q in r.split(8, dim=1):
            t = q - _wilson(_net(q, Ws, side).reshape(side, side, 2, -1), U, -0.10).reshape(q.shape)
            part = ((t.abs() ** 2).sum(0) / (q.abs() ** 2).sum(0)).sum() / c["k"]
            part.backward()
            loss += float(part)
        return {"loss": loss, "grad": torch.cat([w.grad.reshape(-1) for w in Ws]).cpu().numpy()}
    if kind == "solve":
        b = _rhs(c, seed)
        if c["op"] == "wilson":
            U = torch.tensor(_wilson_links(side), device="cuda")
            n = 2 * side * side
            if n > 8192:
                return None
            A = _wilson(torch.eye(n, dtype=torch.complex128, device="cuda").reshape(side, side, 2, n), U, _mass(c))
            return torch.linalg.solve(A.reshape(n, n), b)
        w, V = np.linalg.eigh(_second_difference(side))
        V, w = torch.tensor(V, device="cuda"), torch.tensor(w, device="cuda")
        q = torch.einsum("ai,abk,bj->ijk", V, b.reshape(side, side, -1), V)
        q = q / (w[:, None] + w[None, :])[:, :, None]
        return torch.einsum("ai,ijk,bj->abk", V, q, V).reshape(b.shape)
    if kind == "apply" and c["level"] == 1:
        u = _rhs(c, seed)
        if c["op"] == "wilson":
            return _wilson(u.reshape(side, side, 2, -1), torch.tensor(_wilson_links(side), device="cuda"),
                           _mass(c)).reshape(u.shape)
        return _laplace(u.reshape(side, side, -1)).reshape(u.shape)
    return None
