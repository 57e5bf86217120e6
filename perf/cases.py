"""Performance cases: what a user of this library has it do, through its public calls.

Each case is a dict of plain values.  listed() gives the fixed ones, draw(rng) one more of the same
ranges; prepare() makes what the user's program holds before the call, run() is one pass through the
public entry points, work() the bytes and operations that the pass cannot do without, exact() the same
outputs from plain NumPy in 64 bits.

Kinds:
  run       mctrg_run on a context set up once: trajectories of one lattice, per-trajectory results
            and the estimate read back to the host (the framework's main call)
  batch     mctrg_batch_run: jobs of uneven L and chi in one call, their set-up included
  serve     a server that holds no state between jobs but its workers: jobs submitted together and
            waited for, their set-up included
  hotrg     mctrg_hotrg_run: Monte Carlo HOTRG trajectories
  svd       the batched SVD alone (values and the leading right vectors), by route
  contract  the plaquette contraction alone, by precision
"""
import math
import os
import tempfile

import numpy as np
import torch

from paper_1710_03757_gb300 import mctrg

PRECISIONS = {"fp64": mctrg.MCTRG_FP64, "fp64tc": mctrg.MCTRG_FP64TC, "tf32x3": mctrg.MCTRG_TF32X3}
ROUTES = {"auto": mctrg.SVD_AUTO, "bidiag": mctrg.SVD_BIDIAG, "band": mctrg.SVD_BAND}


def listed():
    return [
        # one request's worth of trajectories on a small lattice: launches and their gaps, 16 x 16 matrices
        {"name": "run-L8-chi4", "kind": "run", "L": 8, "chi": 4, "beta": 0.44, "h": 0.0, "n": 16,
         "precision": "fp64", "route": "auto"},
        # a small lattice of the serving mix, 64 x 64 matrices in quantity
        {"name": "run-L16-chi8", "kind": "run", "L": 16, "chi": 8, "beta": 0.44, "h": 0.0, "n": 256,
         "precision": "fp64", "route": "auto"},
        # the headline chi with default options: 256 x 256 matrices, plain FP64
        {"name": "run-L32-chi16", "kind": "run", "L": 32, "chi": 16, "beta": 0.44, "h": 0.0, "n": 64,
         "precision": "fp64", "route": "auto"},
        # the same trajectories with both tensor-core options on
        {"name": "run-L32-chi16-fp64tc-band", "kind": "run", "L": 32, "chi": 16, "beta": 0.44, "h": 0.0, "n": 64,
         "precision": "fp64tc", "route": "band"},
        # towards the headline lattice, as far as results stay comparable to 1e-9: levels of up to 2048 matrices
        {"name": "run-L64-chi16", "kind": "run", "L": 64, "chi": 16, "beta": 0.44, "h": 0.0, "n": 32,
         "precision": "fp64", "route": "auto"},
        # a chi that is no power of two, in a field: 144 x 144 matrices, ragged tiles
        {"name": "run-L16-chi12-h", "kind": "run", "L": 16, "chi": 12, "beta": 0.40, "h": 0.05, "n": 48,
         "precision": "fp64", "route": "auto"},
        # a large chi of the uneven mix: 576 x 576 matrices, few of them at a time
        {"name": "run-L16-chi24", "kind": "run", "L": 16, "chi": 24, "beta": 0.44, "h": 0.0, "n": 8,
         "precision": "fp64", "route": "auto"},
        # jobs of uneven L and chi in one call, the launch geometry kept from earlier ones
        {"name": "batch-16-jobs", "kind": "batch", "jobs": 16, "Lmax": 32, "chimax": 16, "nmax": 24,
         "precision": "fp64"},
        # a burst of small requests to a server
        {"name": "serve-64-jobs", "kind": "serve", "jobs": 64, "Lmax": 32, "chimax": 8, "nmax": 16},
        # the other coarse-graining scheme
        {"name": "hotrg-L16-chi8", "kind": "hotrg", "L": 16, "chi": 8, "beta": 0.44, "h": 0.0, "n": 16},
        # the batched SVD of level matrices alone, leading vectors for a truncation
        {"name": "svd-n256", "kind": "svd", "route": "bidiag", "size": 256, "batch": 304, "vec": 16},
        # the contraction alone, FP64-accurate on the tensor cores
        {"name": "contract-n256-fp64tc", "kind": "contract", "D": 16, "K": 256, "batch": 512, "precision": "fp64tc"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above; never more work than the largest listed one."""
    kind = rng.choice(["run", "run", "run", "run", "batch", "serve", "hotrg", "svd", "svd", "contract", "contract"])
    if kind == "run":
        while True:
            # the disordered side and the critical point, chi >= 4: in the ordered phase, and at chi = 2, near-
            # degenerate kept and dropped values leave a trajectory's value to the rounding of the basis
            c = {"kind": kind, "L": rng.choice([8, 16, 32, 64]), "chi": rng.choice([4, 5, 6, 8, 10, 12, 16, 20, 24]),
                 "beta": round(rng.uniform(0.30, 0.46), 3), "h": rng.choice([0.0, 0.0, 0.01, 0.05]),
                 "precision": rng.choice(["fp64", "fp64", "fp64tc", "tf32x3"]), "route": "auto"}
            if c["precision"] == "fp64tc":
                c["route"] = "band"
            levels = _distinct_levels(c["L"], c["chi"])
            most = int(min(4000, 4.0e10 / (sum(N * (n ** 3 + 3e5) for N, n, _, _ in levels) + 1e5)))
            if levels and most >= 1:         # a lattice that chi holds exactly has nothing to sample
                c["n"] = _log_int(rng, 1, most)
                return c
    if kind == "batch":
        return {"kind": kind, "jobs": rng.randint(4, 16), "Lmax": rng.choice([16, 32]), "chimax": rng.choice([8, 12, 16]),
                "nmax": rng.randint(4, 24), "precision": rng.choice(["fp64", "fp64tc"])}
    if kind == "serve":
        return {"kind": kind, "jobs": rng.randint(8, 64), "Lmax": rng.choice([8, 16, 32]), "chimax": rng.choice([4, 8]),
                "nmax": rng.randint(4, 16)}
    if kind == "hotrg":
        return {"kind": kind, "L": rng.choice([4, 8, 16]), "chi": rng.choice([3, 4, 5, 6, 8]),
                "beta": round(rng.uniform(0.30, 0.46), 3), "h": rng.choice([0.0, 0.05]), "n": _log_int(rng, 1, 16)}
    if kind == "svd":
        route = rng.choice(["bidiag", "bidiag", "band", "jacobi"])
        size = {"band": 8 * rng.randint(8, 32), "jacobi": _log_int(rng, 8, 128), "bidiag": _log_int(rng, 20, 600)}[route]
        batch = _log_int(rng, 1, max(1, min(2000, int((5e8 if route == "jacobi" else 5e9) / size ** 3))))
        return {"kind": kind, "route": route, "size": size, "batch": batch,
                "vec": 0 if route == "jacobi" else rng.choice([0, 4, 8, 16])}
    prec = rng.choice(["fp64", "fp64tc"])
    D = rng.randint(4, 24)
    K = rng.choice([64, 128, 192, 256, 576]) if prec == "fp64tc" else rng.randint(4, 24) ** 2
    return {"kind": kind, "D": D, "K": K, "batch": _log_int(rng, 1, max(1, int(8e9 / (D ** 4 * K + 1e5)))),
            "precision": prec}


# ---- inputs ----------------------------------------------------------------------------------------
class _Context:
    """A context with its lattice set up, released with the object."""

    def __init__(self, case, options):
        self.handle = mctrg.mctrg_create(options)
        status = mctrg.mctrg_init_lattice(self.handle, case["beta"], case["h"], case["L"], case["chi"])
        if status != mctrg.MCTRG_OK:
            raise RuntimeError("mctrg_init_lattice: " + mctrg.mctrg_strerror(status))

    def __del__(self):
        mctrg.mctrg_destroy(self.handle)


_cache = []


def _launch_cache():
    """The file in which this process keeps the batch runs' launch geometry."""
    if not _cache:
        _cache.append(tempfile.TemporaryDirectory())
    return os.path.join(_cache[0].name, "geometry")


class _Server:
    def __init__(self):
        self.handle = mctrg.mctrg_server_create()

    def __del__(self):
        mctrg.mctrg_server_destroy(self.handle)


def _jobs(case, seed):
    """(beta, h, L, chi, n, seed, first) of an uneven job list; sizes and couplings vary with the seed only
    in their couplings, so that every seed has the same work."""
    shape = np.random.default_rng(case["jobs"] * 1000 + case["nmax"])
    inputs = np.random.default_rng(seed)
    Ls = [v for v in (4, 8, 16, 32) if v <= case["Lmax"]]
    chis = [v for v in (4, 8, 12, 16) if v <= case["chimax"]]
    out = []
    for _ in range(case["jobs"]):
        L, chi = int(shape.choice(Ls)), int(shape.choice(chis))
        n = int(shape.integers(2, case["nmax"] + 1))
        out.append((float(inputs.uniform(0.30, 0.46)), float(inputs.choice([0.0, 0.05])), L, chi, n,
                    int(inputs.integers(1, 1 << 40)), 0))
    return out


def _level_like(size, batch, seed):
    """Matrices with the spectra of level matrices: smooth decay over some fourteen decades."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)
    a = torch.randn(batch, size, size, generator=g, device="cuda", dtype=torch.float64)
    b = torch.randn(batch, size, size, generator=g, device="cuda", dtype=torch.float64)
    s = 10.0 ** (-14.0 * torch.arange(size, device="cuda", dtype=torch.float64) / size)
    return torch.bmm(a * s, b) / size


def _halves_products(D, K, batch, seed):
    """X and Yt of a plaquette: rows that decay over a few decades, as products of reweighted halves do."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)
    n = D * D
    rows = 10.0 ** (-4.0 * torch.arange(n, device="cuda", dtype=torch.float64) / n)
    make = lambda: torch.randn(batch, n, K, generator=g, device="cuda", dtype=torch.float64) * rows[None, :, None]  # noqa: E731
    return make(), make()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "run":
        opts = mctrg.make_options(precision=PRECISIONS[case["precision"]], svd=ROUTES[case["route"]])
        n = case["n"]
        return {"case": case, "ctx": _Context(case, opts), "seed": int(seed), "lnabs": np.zeros(n),
                "sign": np.zeros(n, np.int8), "flags": np.zeros(n, np.uint8)}
    if kind == "batch":
        jobs = _jobs(case, seed)
        n = sum(j[4] for j in jobs)
        opts = mctrg.make_options(precision=PRECISIONS[case["precision"]], autotune_cache=_launch_cache())
        return {"case": case, "jobs": jobs, "opts": opts,
                "lnabs": np.zeros(n), "sign": np.zeros(n, np.int8), "flags": np.zeros(n, np.uint8)}
    if kind == "serve":
        return {"case": case, "jobs": _jobs(case, seed), "server": _Server()}
    if kind == "hotrg":
        n = case["n"]
        return {"case": case, "opts": mctrg.mctrg_options_default(), "seed": int(seed), "lnabs": np.zeros(n),
                "sign": np.zeros(n, np.int8), "flags": np.zeros(n, np.uint8)}
    if kind == "svd":
        n, b, v = case["size"], case["batch"], case["vec"]
        return {"case": case, "M": _level_like(n, b, seed),
                "sigma": torch.zeros(b, n, device="cuda", dtype=torch.float64),
                "vt": torch.zeros(b, v, n, device="cuda", dtype=torch.float64) if v else None}
    X, Yt = _halves_products(case["D"], case["K"], case["batch"], seed)
    n = case["D"] ** 2
    return {"case": case, "X": X, "Yt": Yt, "M": torch.zeros(case["batch"], n, n, device="cuda", dtype=torch.float64)}


# ---- one pass --------------------------------------------------------------------------------------
def _ok(status, what):
    if status not in (mctrg.MCTRG_OK, mctrg.MCTRG_EDOMAIN):
        raise RuntimeError(what + ": " + mctrg.mctrg_strerror(status))


def _estimate(est):
    # not the standard error: it is the spread of lnabsZ (returned whole), which at small beta is that of last digits
    return {"ln_mean_Z": est.ln_mean_Z, "ess": est.ess, "n_negative": est.n_negative, "n_flagged": est.n_flagged}


def _fix_signs(vt):
    """Each vector with its largest entry positive (a singular vector's sign is free)."""
    at = vt.abs().argmax(dim=-1, keepdim=True)
    return vt * vt.gather(-1, at).sign()


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "run":
        status, est = mctrg.mctrg_run(state["ctx"].handle, case["n"], state["seed"], 0, state["lnabs"], state["sign"],
                                      state["flags"])
        _ok(status, "mctrg_run")
        return {"lnabsZ": state["lnabs"], "sign": state["sign"], "flags": state["flags"], "estimate": _estimate(est)}
    if kind == "batch":
        status, ests = mctrg.mctrg_batch_run(state["jobs"], state["opts"], state["lnabs"], state["sign"], state["flags"])
        _ok(status, "mctrg_batch_run")
        return {"lnabsZ": state["lnabs"], "sign": state["sign"], "flags": state["flags"],
                "ln_mean_Z": np.array([e.ln_mean_Z for e in ests])}
    if kind == "serve":
        server = state["server"].handle
        ids = []
        for beta, h, L, chi, n, seed, _ in state["jobs"]:
            status, job = mctrg.mctrg_server_submit(server, beta, h, L, chi, 0.0, n, seed)
            _ok(status, "mctrg_server_submit")
            ids.append(job)
        ests = []
        for job in ids:
            status, est, _ = mctrg.mctrg_server_wait(server, job, 60.0)
            _ok(status, "mctrg_server_wait")
            ests.append(est)
        return {"n": np.array([e.n for e in ests]), "ln_mean_Z": np.array([e.ln_mean_Z for e in ests]),
                "ess": np.array([e.ess for e in ests])}
    if kind == "hotrg":
        status, est = mctrg.mctrg_hotrg_run(state["opts"], case["L"], case["chi"], case["n"], state["seed"],
                                            beta=case["beta"], h=case["h"], lnabsZ=state["lnabs"], sign=state["sign"],
                                            flags=state["flags"])
        _ok(status, "mctrg_hotrg_run")
        return {"lnabsZ": state["lnabs"], "sign": state["sign"], "flags": state["flags"], "estimate": _estimate(est)}
    if kind == "svd":
        call = {"band": mctrg.mctrg_svd_band_batched, "bidiag": mctrg.mctrg_svd_bidiag_batched,
                "jacobi": mctrg.mctrg_svd_batched}[case["route"]]
        _ok(call(state["M"], state["sigma"], state["vt"]), "svd")
        if state["vt"] is None:
            return {"sigma": state["sigma"]}
        return {"sigma": state["sigma"], "vt": _fix_signs(state["vt"])}
    _ok(mctrg.mctrg_contract_batched(state["X"], state["Yt"], state["M"], PRECISIONS[case["precision"]]), "contract")
    return {"M": state["M"]}


# ---- floors ----------------------------------------------------------------------------------------
def _distinct_levels(L, chi):
    """(tensors, matrix side, parents' leg, kept) of the levels that every trajectory splits on its own: those
    after the first one that samples, where the Ising lattice's matrices, of ranks 2, 4, 4, 16, 16, 256, pass chi."""
    ranks = [2, 4, 4, 16, 16]
    levels, D, parent, sampled = [], 2, 2, False
    for k in range(2 * int(math.log2(L))):
        n = D * D
        rank = ranks[k] if not sampled and k < len(ranks) else n
        if sampled:
            levels.append((L * L >> k, n, parent, min(chi, n)))
        sampled = sampled or rank > chi
        parent, D = D, min(chi, rank)
    return levels


def _trg_flops(L, chi, n_traj):
    total = 0.0
    for N, n, d, kc in _distinct_levels(L, chi):
        total += N * (8.0 / 3.0 * n ** 3 + 4.0 * n * n * kc + 2.0 * n * n * d * d + 4.0 * n * d ** 3 + 4.0 * n * kc)
    return n_traj * (total + 4.0 * chi ** 4)


def work(case):
    """Reduction, kept vectors, plaquette contraction and choice per tensor; bytes of inputs and results."""
    kind = case["kind"]
    if kind == "run":
        return {"bytes": 10.0 * case["n"] + 128, "flops": _trg_flops(case["L"], case["chi"], case["n"])}
    if kind in ("batch", "serve"):
        jobs = _jobs(case, 0)
        return {"bytes": sum(10.0 * j[4] + 128 for j in jobs), "flops": sum(_trg_flops(j[2], j[3], j[4]) for j in jobs)}
    if kind == "hotrg":
        total, Lx, Ly, Dh, Dv = 0.0, case["L"], case["L"], 2, 2
        while Lx * Ly > 1:
            n, kc, N = Dh * Dh, min(case["chi"], Dh * Dh), Lx * Ly // 2
            q = Dh * Dv
            total += N * (4.0 * q ** 3 + 2.0 * n * n * Dv * Dv + 8.0 / 3.0 * n ** 3 + 4.0 * n * n * kc +
                          2.0 * kc * Dv * Dh * Dh * Dv * (Dh + q) + 2.0 * kc * Dv * kc * Dv * n)
            Lx, Ly, Dh, Dv = Ly // 2, Lx, Dv, kc
        return {"bytes": 10.0 * case["n"] + 128, "flops": case["n"] * total}
    if kind == "svd":
        n, b, v = case["size"], case["batch"], case["vec"]
        return {"bytes": 8.0 * b * (n * n + n + v * n), "flops": b * (8.0 / 3.0 * n ** 3 + 4.0 * n * n * v)}
    n, K, b = case["D"] ** 2, case["K"], case["batch"]
    return {"bytes": 8.0 * b * (2.0 * n * K + n * n), "flops": 2.0 * b * n * n * K}


# ---- the same outputs in plain NumPy ---------------------------------------------------------------
def _philox(seed, traj, level, tensor, t):
    """Philox4x32-10 uniforms (Salmon et al. 2011) for arrays of trajectories and tensors, draw step t."""
    m32 = np.uint64(0xFFFFFFFF)
    traj, tensor = np.broadcast_arrays(np.asarray(traj, np.uint64), np.asarray(tensor, np.uint64))
    c = [np.full(traj.shape, t >> 1, np.uint64), tensor.copy(), np.full(traj.shape, level, np.uint64), traj.copy()]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    lo, hi = (c[2], c[3]) if t & 1 else (c[0], c[1])
    return (((hi << np.uint64(32)) | lo) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _choose(s, chi, uniforms):
    """Kept indices and inclusion rates of chi-subsets with p(e) ~ prod s^2, for rows of spectra s / s_1 (zeros
    already 0): the largest kept index first, by running sums of elementary symmetric polynomials."""
    items, n = s.shape
    w = s * s
    E = np.zeros((n + 1, items, chi + 1))
    E[0, :, 0] = 1.0
    for i in range(1, n + 1):
        E[i] = E[i - 1]
        E[i, :, 1:] += w[:, i - 1, None] * E[i - 1, :, :-1]
    rows, b = np.arange(items), np.full(items, n)
    kept = np.zeros((items, chi), int)
    for t in range(chi):
        j = chi - t
        x = uniforms(t) * E[b, rows, j]
        i = np.argmax(E[:, :, j] > x[None, :], axis=0)
        kept[:, j - 1] = i - 1
        b = i - 1
    e_all = E[n, :, chi]
    rate = np.zeros((items, chi))
    for a in range(chi):
        e = np.zeros((items, chi))
        e[:, 0] = 1.0
        for i in range(n):
            wi = np.where(kept[:, a] == i, 0.0, w[:, i])
            e[:, 1:] += wi[:, None] * e[:, :-1]
        rate[:, a] = w[rows, kept[:, a]] * e[:, chi - 1] / e_all
    return kept, rate


def _split(M, chi, Dn, uniforms):
    """Halves (left, right) and ln s_1 of a stack of matrices; uniforms None keeps every nonzero value."""
    U, s, Vt = np.linalg.svd(M)
    n = M.shape[-1]
    rel = s / s[:, :1]
    rel[rel <= n * 2.0 ** -52] = 0.0
    items = len(M)
    left, right = np.zeros((items, n, Dn)), np.zeros((items, Dn, n))
    few = (rel > 0).sum(axis=1) <= chi
    for which in (np.flatnonzero(few), np.flatnonzero(~few)):
        if not len(which):
            continue
        if few[which[0]]:
            kept = np.tile(np.arange(min(Dn, n)), (len(which), 1))
            st = np.take_along_axis(rel[which], kept, 1)
        else:
            kept, rate = _choose(rel[which], chi, lambda t: uniforms(t)[which])
            st = np.take_along_axis(rel[which], kept, 1) / rate
        k, root = kept.shape[1], np.sqrt(st)
        left[which, :, :k] = np.take_along_axis(U[which], kept[:, None, :], 2) * root[:, None, :]
        right[which, :k, :] = np.take_along_axis(Vt[which], kept[:, :, None], 1) * root[:, :, None]
    return left, right, np.log(s[:, 0])


def _site_tensor(beta, h):
    W = np.array([[math.sqrt(math.cosh(beta)), sg * math.sqrt(math.sinh(beta))] for sg in (1.0, -1.0)])
    return np.einsum("s,sa,sb,sc,sd->abcd", np.exp(beta * h * np.array([1.0, -1.0])), W, W, W, W)


def _matricize(T, odd):
    D = T.shape[1]
    return (T.transpose(0, 2, 3, 4, 1) if odd else T).reshape(len(T), D * D, D * D)


def _plaquette(F3, F4, F2, F1):
    d, D = int(round(math.sqrt(F3.shape[2]))), F3.shape[1]
    X = np.einsum("taij,tbki->tabjk", F3.reshape(-1, D, d, d), F4.reshape(-1, D, d, d)).reshape(-1, D * D, d * d)
    Y = np.einsum("tjmg,tmkd->tdgjk", F2.reshape(-1, d, d, D), F1.reshape(-1, d, d, D)).reshape(-1, D * D, d * d)
    return np.matmul(X, Y.transpose(0, 2, 1)).reshape(-1, D, D, D, D)


def _trg(beta, h, L, chi, n, seed, first=0):
    """ln|Z~| and sign of Monte Carlo TRG trajectories first .. first + n - 1 (Levin-Nave levels)."""
    T = _site_tensor(beta, h)[None]
    sites = [(x, y) for y in range(L) for x in range(L)]
    a1, a2 = (1, 0), (0, 1)
    lnacc, shared = np.zeros(n), True
    traj = np.arange(first, first + n)
    for level in range(2 * int(math.log2(L))):
        b1, b2 = (a1[0] + a2[0], a1[1] + a2[1]), (a2[0] - a1[0], a2[1] - a1[1])
        even = {((i * b1[0] + j * b2[0]) % L, (i * b1[1] + j * b2[1]) % L) for i in range(L) for j in range(L)}
        index = {p: t for t, p in enumerate(sites)}
        odd = np.array([p not in even for p in sites])
        new = [p for p in sites if p in even]
        at = lambda p, v: index[((p[0] + v[0]) % L, (p[1] + v[1]) % L)]  # noqa: E731
        parents = np.array([[index[p], at(p, a1), at(p, a2), at(p, b1)] for p in new])
        N, D = len(sites), T.shape[-1]
        nn = D * D
        if shared:
            s = np.linalg.svd(np.concatenate([_matricize(T, False), _matricize(T, True)]), compute_uv=False)
            rank = int((s / s[:, :1] > nn * 2.0 ** -52).sum(axis=1).max())
            Dn = max(1, min(chi, rank))
            if rank <= chi:
                (La, Ra, sa), (Lb, Rb, sb) = (_split(_matricize(T, o), chi, Dn, None) for o in (False, True))
                lnacc += (N // 2) * (sa[0] + sb[0])
                T = _plaquette(Ra, Rb, Lb, La)
                sites, a1, a2 = new, b1, b2
                continue
            T = np.broadcast_to(T, (n * N,) + T.shape[1:])
            shared = False
        else:
            Dn = min(chi, nn)
        odds, tens, trs = np.tile(odd, n), np.tile(np.arange(N), n), np.repeat(traj, N)
        M = np.where(odds[:, None, None], _matricize(T, True), _matricize(T, False))
        left, right, ln1 = _split(M, chi, Dn, lambda t, lv=level: _philox(seed, trs, lv, tens, t))
        lnacc += ln1.reshape(n, N).sum(axis=1)
        pick = (np.arange(n)[:, None, None] * N + parents[None]).reshape(-1, 4)
        T = _plaquette(right[pick[:, 0]], right[pick[:, 1]], left[pick[:, 2]], left[pick[:, 3]])
        sites, a1, a2 = new, b1, b2
    tr = np.broadcast_to(np.einsum("tabab->t", T), (n,))
    return lnacc + np.log(np.abs(tr)), np.sign(tr)


def _hotrg(beta, h, L, chi, n, seed):
    """ln|Z~| and sign of Monte Carlo HOTRG trajectories: rows merged in pairs, each merged bond truncated by a
    random projector from its Gram matrix, the lattice reflected after every step."""
    T = np.broadcast_to(_site_tensor(beta, h), (n, L, L, 2, 2, 2, 2))      # [trajectory][y][x][l][u][r][d]
    lnacc = np.zeros(n)
    for step in range(2 * int(math.log2(L))):
        Ly, Lx, Dh, Dv = T.shape[1], T.shape[2], T.shape[3], T.shape[4]
        m, Lj = Dh * Dh, Ly // 2
        kc, N = min(chi, m), Lx * (Ly // 2)
        M = np.einsum("...aurk,...bksd->...abursd", T[:, 0::2], T[:, 1::2], optimize=True).reshape(n * N, m, Dv, m, Dv)
        R = M.transpose(0, 3, 1, 2, 4).reshape(n * N, m, -1)
        lam, V = np.linalg.eigh(np.matmul(R, R.transpose(0, 2, 1)))
        lam, V = lam[:, ::-1], V[:, :, ::-1]
        rel = np.sqrt(np.where(lam > m * 2.0 ** -52 * lam[:, :1], lam / lam[:, :1], 0.0))
        F = np.zeros((n * N, m, kc))
        few = (rel > 0).sum(axis=1) <= chi
        trs, bonds = np.repeat(np.arange(n), N), np.tile(np.arange(N), n)
        for which in (np.flatnonzero(few), np.flatnonzero(~few)):
            if not len(which):
                continue
            if few[which[0]]:
                F[which] = V[which][:, :, :kc] * (rel[which][:, None, :kc] > 0)
            else:
                kept, rate = _choose(rel[which], chi, lambda t: _philox(seed, trs[which], step, bonds[which], t))
                F[which] = np.take_along_axis(V[which], kept[:, None, :], 2) / np.sqrt(rate)[:, None, :]
        lnacc += 0.5 * np.log(lam[:, 0]).reshape(n, N).sum(axis=1)
        FL = np.roll(F.reshape(n, Lj, Lx, m, kc), 1, axis=2).reshape(n * N, m, kc)
        P = np.matmul(FL.transpose(0, 2, 1), M.reshape(n * N, m, -1)).reshape(n * N, kc, Dv, m, Dv)
        new = np.einsum("taurd,trb->taubd", P, F, optimize=True) / np.sqrt(lam[:, 0])[:, None, None, None, None]
        T = new.reshape(n, Lj, Lx, kc, Dv, kc, Dv).transpose(0, 2, 1, 4, 3, 6, 5)
    tr = np.einsum("tabab->t", T[:, 0, 0])
    return lnacc + np.log(np.abs(tr)), np.sign(tr)


def _exact_estimate(lnabs, sign):
    top = lnabs.max()
    x = sign * np.exp(lnabs - top)
    return {"ln_mean_Z": float(top + math.log(x.mean())) if x.mean() > 0 else None,
            "ess": float(x.sum() ** 2 / (x * x).sum()), "n_negative": None, "n_flagged": None}


def _seconds(L, chi, n):
    """About how long _trg takes (measured: a 256 x 256 SVD 25 ms, the choice 0.2 us per value and kept index)."""
    return n * sum(N * (1.5e-9 * s ** 3 + 1e-4 + 8e-8 * s * chi * chi) for N, s, _, _ in _distinct_levels(L, chi))


def exact(case, seed):
    kind = case["kind"]
    if kind == "run":
        if _seconds(case["L"], case["chi"], case["n"]) > 9 or case["precision"] == "tf32x3":
            return None
        lnabs, sign = _trg(case["beta"], case["h"], case["L"], case["chi"], case["n"], int(seed))
        return {"lnabsZ": lnabs, "sign": None, "flags": None, "estimate": _exact_estimate(lnabs, sign)}
    if kind in ("batch", "serve"):
        jobs = _jobs(case, seed)
        if sum(_seconds(j[2], j[3], j[4]) for j in jobs) > 9:
            return None
        every = [_trg(*j) for j in jobs]
        ests = [_exact_estimate(*e) for e in every]
        if any(e["ln_mean_Z"] is None for e in ests):
            return None
        column = lambda k: np.array([e[k] for e in ests])  # noqa: E731
        if kind == "serve":
            return {"n": None, "ln_mean_Z": column("ln_mean_Z"), "ess": column("ess")}
        return {"lnabsZ": np.concatenate([e[0] for e in every]), "sign": None, "flags": None,
                "ln_mean_Z": column("ln_mean_Z")}
    if kind == "hotrg":
        lnabs, sign = _hotrg(case["beta"], case["h"], case["L"], case["chi"], case["n"], int(seed))
        return {"lnabsZ": lnabs, "sign": None, "flags": None, "estimate": _exact_estimate(lnabs, sign)}
    if kind == "svd":
        M = _level_like(case["size"], case["batch"], seed)
        if case["batch"] * (1.5e-9 * case["size"] ** 3 + 1e-4) > 12:
            return None
        _, s, Vt = np.linalg.svd(M.cpu().numpy())
        out = {"sigma": torch.from_numpy(s)}
        if case["vec"]:
            out["vt"] = _fix_signs(torch.from_numpy(Vt[:, :case["vec"]].copy()))
        return out
    X, Yt = _halves_products(case["D"], case["K"], case["batch"], seed)
    return {"M": torch.bmm(X, Yt.transpose(1, 2))}
