"""The workloads this library is measured on, through its public entry points.

A case is one shape of one call: the three MTTKRPs of a tensor, ALS sweeps, a GD
step, a batched sweep of many jobs, the build of the CSR copies, a sweep of the
joint ratings + reviews model.  ``listed()`` names twelve of them, ``draw(rng)``
gives more of the same ranges, ``prepare`` makes what a user's program has in
hand (tensor, factors, handle), ``run`` makes one pass, ``work`` counts the bytes
and operations a pass cannot do without, and ``exact`` is the same pass in plain
64-bit torch, written from the method's definitions.

Keys of a case: op; dist (how the coordinates are drawn: "uniform", "zipf" with
exponents s0, s1, s2, "pa" preferential attachment); I, J, K, nnz; R; dtype
(factor storage, "f32" or "bf16"); values ("uniform", "lognormal", "cp").
"""
import math

import numpy as np
import torch

from paper_1406_4519_gb300 import dfacto, synth

_DT = {"f32": (dfacto.F32, torch.float32, 4), "bf16": (dfacto.BF16, torch.bfloat16, 2)}


def _case(op, dist, dims, nnz, R, dtype="f32", values="uniform", s=(0.0, 0.0, 0.0), **more):
    c = {"op": op, "dist": dist, "I": dims[0], "J": dims[1], "K": dims[2], "nnz": nnz, "R": R,
         "dtype": dtype, "values": values, "s0": s[0], "s1": s[1], "s2": s[2]}
    c.update(more)
    return c


def listed():
    z50 = ([1000000, 500000, 200000], 50000000)
    return [
        # The headline workload's hot path: every mode's MTTKRP of a large power-law
        # tensor whose factors fit the L2 (the inside of ALS and GD).
        dict(_case("mttkrp", "zipf", *z50, 32, values="lognormal", s=(1.2, 1.2, 1.2)),
             name="mttkrp_zipf50M_r32"),
        # The 1.2B-nonzero review-tensor workload (rank 10: not a multiple of four)
        # scaled by 0.05, the replica its profiles are taken on.
        dict(_case("mttkrp", "zipf", [325000, 125000, 75000], 60000000, 10, values="lognormal",
                   s=(1.1, 1.3, 1.2)), name="mttkrp_zipf60M_r10"),
        # The largest job of the batched/served mix alone: uniform coordinates (most
        # fibers hold one nonzero) and BF16 factors.
        dict(_case("mttkrp", "uniform", [200000, 150000, 100000], 5000000, 16, "bf16"),
             name="mttkrp_uniform5M_r16_bf16"),
        # The smallest call: the 10,000-nonzero configuration, five sweeps from given
        # factors with the fit read after each; latency and launches.
        dict(_case("als", "uniform", [200, 150, 100], 10000, 10, sweeps=5), name="als_uniform10k_r10"),
        # The headline: one sweep of an ALS loop on the planted rank-32 tensor.
        dict(_case("als", "zipf", *z50, 32, values="cp", s=(1.2, 1.2, 1.2), sweeps=0),
             name="als_zipf50M_r32"),
        # The paper's largest synthetic set (Table 5): ten million indices per mode and
        # two nonzeros per index, so the dense row passes outweigh the nonzeros.
        dict(_case("als", "pa", [10000000] * 3, 20000000, 10, sweeps=0), name="als_pa2I_1e7_r10"),
        # The gradient method on the headline tensor: three gradients, line search, update.
        dict(_case("gd", "zipf", *z50, 32, values="cp", s=(1.2, 1.2, 1.2)),
             name="gd_zipf50M_r32"),
        # The gradient method on a middle set of the paper's Table 4.
        dict(_case("gd", "pa", [100000] * 3, 1000000, 10), name="gd_pa1M_1e5_r10"),
        # A quarter-size batch of the batched configuration with BF16 factors (as the
        # server runs them): one graph-replayed sweep of 48 uneven jobs.
        dict(_case("batch", "uniform", [0, 0, 0], 0, 0, "bf16", jobs=48, specs=14064523),
             name="batch_48jobs_bf16"),
        # A new tensor: COO to three CSR copies, at the headline size ...
        dict(_case("build", "zipf", *z50, 32, values="lognormal", s=(1.2, 1.2, 1.2)),
             name="build_zipf50M"),
        # ... and at the size of a served request.
        dict(_case("build", "uniform", [60000, 20000, 5000], 500000, 16, "bf16"),
             name="build_uniform500k"),
        # Ratings + reviews (Appendix F): one sweep of row solves from start factors.
        dict(_case("joint", "zipf", [100000, 50000, 20000], 0, 16, ratings=2000000, words=4),
             name="joint_als_2M_r16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["mttkrp", "mttkrp", "mttkrp", "als", "als", "gd", "batch", "build", "joint"])
    R = rng.choice([1, 3, 4, 7, 8, 10, 12, 13, 16, 16, 20, 24, 30, 32, 32, 40, 64])
    dtype = rng.choice(["f32", "f32", "bf16"])
    if op == "batch":
        return _case("batch", "uniform", [0, 0, 0], 0, 0, dtype, jobs=rng.randint(3, 40),
                     specs=rng.randrange(1 << 30))
    if op == "joint":
        users = _log_int(rng, 300, 100000)
        items = _log_int(rng, 200, 50000)
        return _case("joint", "zipf", [users, items, _log_int(rng, 150, 20000)], 0,
                     rng.choice([8, 10, 16, 32]), dtype,
                     ratings=min(_log_int(rng, 3000, 1500000), users * items // 20),
                     words=rng.randint(1, 6))
    dist = rng.choice(["zipf", "zipf", "uniform", "pa"])
    nnz = _log_int(rng, 10000, min(4.0e7, 1.2e9 / R))
    s = (0.0, 0.0, 0.0)
    if dist == "zipf":  # power-law modes with indices to spare for unique coordinates
        dims = [_log_int(rng, max(1000, nnz ** 0.5 * 8), max(4000, nnz ** 0.5 * 150)) for _ in range(3)]
        s = tuple(round(rng.uniform(1.05, 1.25), 2) for _ in range(3))
        values = rng.choice(["lognormal", "uniform"])
    else:
        nnz = min(nnz, 10000000)
        lo = max(50, (4 * nnz) ** (1 / 3))
        dims = [_log_int(rng, lo, max(2 * lo, min(4.0e6, 2 * nnz))) for _ in range(3)]
        values = "uniform"
    more = {"sweeps": 0} if op == "als" else {}
    return _case(op, dist, dims, nnz, R, dtype, values, s, **more)


def _dims(c):
    return [c["I"], c["J"], c["K"]]


def _tensor(c, seed):
    dims = _dims(c)
    if c["dist"] == "zipf":
        return synth.zipf_tensor(dims, c["nnz"], [c["s0"], c["s1"], c["s2"]], seed, "cuda",
                                 values=c["values"], R_true=min(c["R"], 32))
    if c["dist"] == "pa":
        return synth.preferential_attachment_tensor(dims, c["nnz"], seed, "cuda")
    return synth.uniform_tensor(dims, c["nnz"], seed, "cuda")


def _coo(c, seed):
    """A tensor whose number of fibers does not depend on the seed (the build returns
    arrays of that length): one set of coordinates, its labels rotated along every axis,
    the order shuffled and the values drawn by the seed."""
    idx, val = _tensor(c, 14064521)
    g = synth.generator(seed, "cuda")
    order = torch.randperm(val.numel(), generator=g, device="cuda")
    shift = torch.randint(0, 1 << 30, (3, 1), generator=g, device="cuda")
    dims = torch.tensor(_dims(c), device="cuda")[:, None]
    idx = ((idx[:, order] + shift) % dims).to(torch.int32).contiguous()
    return idx, torch.exp(torch.randn(val.numel(), generator=g, device="cuda"))


def _factors(c, dims, R, seed):
    F = synth.normal_factors(dims, R, seed + 101, "cuda")
    if c["op"] == "joint":  # the scale of the planted ratings and reviews
        F = [f * R ** -0.5 for f in F]
    return [f.to(_DT[c["dtype"]][1]) for f in F]


def _specs(c):
    return synth.batch_job_specs(c["jobs"], c["specs"])


def _joint_inputs(c, seed):
    return synth.joint_ratings_reviews(c["I"], c["J"], c["K"], c["ratings"], c["words"], c["R"],
                                       seed, "cuda")


_JOINT_LAMBDA, _JOINT_MU = 0.1, 0.5


def prepare(c, seed):
    op, (code, tdt, _) = c["op"], _DT[c["dtype"]]
    st = {"op": op, "case": c}
    if op == "batch":
        st["jobs"] = []
        specs = _specs(c)
        for k, s in enumerate(specs):
            idx, val = synth.uniform_tensor(s["dims"], s["nnz"], seed * 4099 + k, "cuda")
            t = dfacto.Tensor(idx, val, s["dims"], rank=s["R"], factor_dtype=code)
            t.set_factors(_factors(c, s["dims"], s["R"], seed * 4099 + k))
            st["jobs"].append(t)
        st["batch"] = dfacto.Batch(st["jobs"])
        # factors come back into one buffer per mode, the jobs one after another
        st["out"] = [torch.empty(sum(s["dims"][m] * s["R"] for s in specs), dtype=tdt, device="cuda")
                     for m in range(3)]
        return st
    if op == "joint":
        yidx, yval, idx, val = _joint_inputs(c, seed)
        t = dfacto.Tensor(idx, val, _dims(c), rank=c["R"], factor_dtype=code, lambda_reg=_JOINT_LAMBDA)
        st["start"] = _factors(c, _dims(c), c["R"], seed)
        t.set_ratings(yidx, yval, _JOINT_MU)
        st["t"] = t
    else:
        idx, val = _coo(c, seed) if op == "build" else _tensor(c, seed)
        if op == "build":
            st["coo"] = (idx, val)
            return st
        t = dfacto.Tensor(idx, val, _dims(c), rank=c["R"], factor_dtype=code)
        st["start"] = _factors(c, _dims(c), c["R"], seed)
        t.set_factors(st["start"])
        st["t"] = t
    st["out"] = [torch.empty(d, c["R"], dtype=torch.float32 if op == "mttkrp" else tdt, device="cuda")
                 for d in _dims(c)]
    return st


def _read_factors(t, out):
    return [dfacto.dfacto_get_factors(t.h, m, out[m]) for m in range(3)]


class _Owned:
    """n elements of a handle's device memory that keep the handle alive (torch holds on
    to the object whose memory it views)."""

    def __init__(self, owner, ptr, n, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (int(n),), "typestr": typestr,
                                         "data": (int(ptr), False), "version": 2}


def _csr(t, mode):
    v = dfacto.dfacto_get_csr(t.h, mode)
    return [torch.as_tensor(_Owned(t, ptr, n, typestr), device="cuda")
            for ptr, n, typestr in ((v.fiber_ptr, v.dim_o + 1, "<i8"), (v.fiber_idx, v.nfib, "<i4"),
                                    (v.nz_ptr, v.nfib + 1, "<i8"), (v.nz_idx, v.nnz, "<i4"),
                                    (v.nz_val, v.nnz, "<f4"))]


def _f32(x):
    # fits, losses and weights are FP64 combinations of FP32 sums over the
    # nonzeros: their meaningful digits are those of FP32
    return np.asarray(x, dtype=np.float32)


def run(st):
    op, c = st["op"], st["case"]
    if op == "mttkrp":
        return [st["t"].mttkrp(m, st["out"][m]) for m in range(3)]
    if op == "als":
        t = st["t"]
        if c["sweeps"]:  # a whole small request: from the start factors, the fit watched
            t.set_factors(st["start"])
        fits = [t.als_iter()[1] for _ in range(max(1, c["sweeps"]))]
        return {"factors": _read_factors(t, st["out"]), "lambda": _f32(t.lam()),
                "residual": _f32([1.0 - f for f in fits])}
    if op == "gd":
        _, loss, step = st["t"].gd_iter()
        return {"factors": _read_factors(st["t"], st["out"]), "loss": _f32(loss), "step": _f32(step)}
    if op == "joint":
        st["t"].set_factors(st["start"])
        obj = st["t"].joint_als_iter()
        return {"factors": _read_factors(st["t"], st["out"]), "objective": _f32(obj)}
    if op == "batch":
        _, fits = st["batch"].als_iter()
        at = [0, 0, 0]
        for t in st["jobs"]:
            for m in range(3):
                n = t.dims[m] * t.rank
                dfacto.dfacto_get_factors(t.h, m, st["out"][m][at[m]:at[m] + n])
                at[m] += n
        return {"factors": st["out"], "residual": _f32([1.0 - f for f in fits])}
    idx, val = st["coo"]
    t = dfacto.Tensor(idx, val, _dims(c), rank=c["R"], factor_dtype=_DT[c["dtype"]][0])
    return [_csr(t, m) for m in range(3)]


def work(c):
    op, s = c["op"], _DT[c["dtype"]][2]

    def mttkrps(dims, nnz, R):  # nonzeros (index and value) once per mode, factors, outputs
        rows = sum(dims)
        return 3 * 8 * nnz + 2 * rows * R * s + 4 * rows * R, 3 * 2 * nnz * R

    if op == "batch":
        b = f = 0
        for j in _specs(c):
            jb, jf = mttkrps(j["dims"], j["nnz"], j["R"])
            b += jb
            f += jf + sum(j["dims"]) * 4 * j["R"] * j["R"]
        return {"bytes": b, "flops": f}
    dims, R = _dims(c), c["R"]
    rows = sum(dims)
    if op == "build":  # COO in; per mode (index, value) per nonzero and row pointers out
        return {"bytes": 16 * c["nnz"] + 3 * 8 * c["nnz"] + 8 * rows, "flops": 0}
    if op == "joint":
        nnz, n = c["ratings"] * c["words"], c["ratings"]
        b, f = mttkrps(dims, nnz, R)
        return {"bytes": b + 2 * 8 * n, "flops": f + 2 * 2 * n * R * R + rows * R ** 3 // 3}
    b, f = mttkrps(dims, c["nnz"], R)
    if op == "mttkrp":
        return {"bytes": b, "flops": f}
    if op == "als":  # N Gamma^-1 and the Gram of the result per row
        k = max(1, c["sweeps"])
        return {"bytes": k * b, "flops": k * (f + rows * 4 * R * R)}
    # gd: the gradients and one more walk for the line search
    return {"bytes": b + 8 * c["nnz"] + rows * R * s, "flops": f + 4 * 2 * c["nnz"] * R + rows * 8 * R * R}


# ---- the same passes in 64 bits ------------------------------------------------

_CHUNK = 1 << 21


def _mttkrp64(idx, val, F, mode):
    """N[o] = sum over the nonzeros of row o of x F_in[in] * F_f[f]."""
    o, i, f = mode, (mode + 1) % 3, (mode + 2) % 3
    order = torch.argsort(idx[o])
    out = torch.zeros(F[o].shape[0], F[o].shape[1], dtype=torch.float64, device="cuda")
    for p in range(0, order.numel(), _CHUNK):
        sel = order[p:p + _CHUNK]
        prod = val[sel].double()[:, None] * F[i][idx[i, sel].long()] * F[f][idx[f, sel].long()]
        rows, count = torch.unique_consecutive(idx[o, sel].long(), return_counts=True)
        ends = torch.cumsum(prod.T.contiguous(), 1)[:, torch.cumsum(count, 0) - 1]
        out.index_add_(0, rows, torch.diff(ends, dim=1, prepend=torch.zeros_like(ends[:, :1])).T)
    return out


def _als64(idx, val, F):
    F = [f.double() for f in F]
    lam = N = None
    for m in range(3):
        i, f = (m + 1) % 3, (m + 2) % 3
        N = _mttkrp64(idx, val, F, m)
        G = (F[f].T @ F[f]) * (F[i].T @ F[i])
        U = torch.linalg.solve(G, N.T).T
        lam = U.norm(dim=0)
        F[m] = U / torch.where(lam > 0, lam, torch.ones_like(lam))
    inner = float(((N * F[2]).sum(0) * lam).sum())
    model = float(lam @ ((F[0].T @ F[0]) * (F[1].T @ F[1]) * (F[2].T @ F[2])) @ lam)
    x2 = float(val.double().square().sum())
    return F, lam, math.sqrt(max(0.0, x2 - 2 * inner + model) / x2)


def _gd64(idx, val, F):
    """One step from F: gradients -N + F Gamma, Armijo backtracking from 1, update."""
    F = [f.double() for f in F]
    G = []
    for m in range(3):
        i, f = (m + 1) % 3, (m + 2) % 3
        G.append(F[m] @ ((F[i].T @ F[i]) * (F[f].T @ F[f])) - _mttkrp64(idx, val, F, m))
    t = [0.0] * 4  # <X, [[A - a GA, B - a GB, C - a GC]]> = sum_k t[k] a^k
    for p in range(0, val.numel(), _CHUNK):
        ix = idx[:, p:p + _CHUNK].long()
        poly = [val[p:p + _CHUNK].double()[:, None]]
        for m in range(3):
            a, g = F[m][ix[m]], G[m][ix[m]]
            low = [q * a for q in poly] + [0.0]
            poly = [low[k] - (poly[k - 1] * g if k else 0.0) for k in range(len(poly) + 1)]
        t = [u + float(q.sum()) for u, q in zip(t, poly)]
    x2 = float(val.double().square().sum())

    def loss(a):
        H = [f - a * g for f, g in zip(F, G)]
        model = float(((H[0].T @ H[0]) * (H[1].T @ H[1]) * (H[2].T @ H[2])).sum())
        return 0.5 * (x2 - 2 * sum(t[k] * a ** k for k in range(4)) + model)

    g2 = sum(float(g.square().sum()) for g in G)
    f0, a = loss(0.0), 1.0
    for _ in range(100):
        if loss(a) <= f0 - 1e-4 * a * g2:
            break
        a *= 0.5
    return [f - a * g for f, g in zip(F, G)], loss(a), a


def _joint64(c, seed):
    yidx, yval, idx, val = _joint_inputs(c, seed)
    F = [f.double() for f in _factors(c, _dims(c), c["R"], seed)]
    R, mu, lam = c["R"], _JOINT_MU, _JOINT_LAMBDA
    eye = torch.eye(R, dtype=torch.float64, device="cuda")
    for m in range(3):
        i, f = (m + 1) % 3, (m + 2) % 3
        H = mu * (F[i].T @ F[i]) * (F[f].T @ F[f]) + lam * eye
        rhs = mu * _mttkrp64(idx, val, F, m)
        if m < 2:
            H = H.repeat(F[m].shape[0], 1, 1)
            own, other = yidx[m].long(), F[1 - m]
            for p in range(0, own.numel(), _CHUNK // 8):
                v = other[yidx[1 - m, p:p + _CHUNK // 8].long()]
                H.index_add_(0, own[p:p + _CHUNK // 8], v[:, :, None] * v[:, None, :])
                rhs.index_add_(0, own[p:p + _CHUNK // 8], v * yval[p:p + _CHUNK // 8, None].double())
            F[m] = torch.linalg.solve(H, rhs[:, :, None])[:, :, 0]
        else:
            F[m] = torch.linalg.solve(H, rhs.T).T
    ix, iy = idx.long(), yidx.long()
    inner = float((val.double() * (F[0][ix[0]] * F[1][ix[1]] * F[2][ix[2]]).sum(1)).sum())
    model = float(((F[0].T @ F[0]) * (F[1].T @ F[1]) * (F[2].T @ F[2])).sum())
    fit = (yval.double() - (F[0][iy[0]] * F[1][iy[1]]).sum(1)).square().sum()
    ridge = sum(float(f.square().sum()) for f in F)
    obj = 0.5 * (float(fit) + mu * (float(val.double().square().sum()) - 2 * inner + model) + lam * ridge)
    return F, obj


def exact(c, seed):
    op = c["op"]
    if op == "joint":
        F, obj = _joint64(c, seed)
        return {"factors": F, "objective": obj}
    if op == "batch":
        out, residual = [[], [], []], []
        for k, s in enumerate(_specs(c)):
            idx, val = synth.uniform_tensor(s["dims"], s["nnz"], seed * 4099 + k, "cuda")
            F, _, r = _als64(idx, val, _factors(c, s["dims"], s["R"], seed * 4099 + k))
            residual.append(r)
            for m in range(3):
                out[m].append(F[m].reshape(-1))
        return {"factors": [torch.cat(o) for o in out], "residual": np.asarray(residual)}
    idx, val = _coo(c, seed) if op == "build" else _tensor(c, seed)
    if op == "build":  # values in (row, fiber, entry) order; indices are whole numbers
        got = []
        for m in range(3):
            order = torch.arange(val.numel(), device="cuda")
            for axis in ((m + 1) % 3, (m + 2) % 3, m):
                order = order[torch.sort(idx[axis, order], stable=True).indices]
            got.append([None, None, None, None, val[order].double()])
        return got
    F = _factors(c, _dims(c), c["R"], seed)
    if op == "mttkrp":
        F = [f.double() for f in F]
        return [_mttkrp64(idx, val, F, m) for m in range(3)]
    if op == "als":
        residual, lam = [], None
        for _ in range(max(1, c["sweeps"])):
            F, lam, r = _als64(idx, val, F)
            residual.append(r)
        return {"factors": F, "lambda": lam, "residual": np.asarray(residual)}
    F, loss, step = _gd64(idx, val, F)
    return {"factors": F, "loss": loss, "step": step}
