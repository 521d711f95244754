"""The work a program has this library do, as timed cases.

Each case is one pass through the public entry points (``vbgs_update``,
``vbgs_elbo``, ``vbgs_reassign``, ``vbgs_render``, ``vbgs_update_batched``,
``vbgs_estep_noalloc``) on the inputs of the repository's own configurations:
mixture points, the room stream, uneven scenes, and the small and ragged sizes
of its tests.  Kinds:

* ``fit``       a mixture fitted from an empty statistics buffer: reset the
                buffer, n_iters CAVI iterations over the points, read the
                statistics back
* ``stream``    one frame of a continual RGB-D stream, after the frames before
                it: n_iters iterations, then the frame's statistics
* ``score``     the per-point ELBO terms of a frame under the streamed posterior
* ``reassign``  Alg. 1's reassign on a frame: the chosen points and components
                and the terms they were ranked on
* ``render``    an image of the streamed posterior at a held-out pose
* ``batched``   uneven scenes in one ``vbgs_update_batched`` call
* ``estep``     the E-step into the caller's device buffers

``exact`` restates the update in 64-bit torch operations, without the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_08499_gb300 import synth, vbgs as V

D, F = 6, 28
WARM = 3          # frames a stream has seen before the timed one
AHEAD = 4         # frames it cycles through from there


def listed():
    return [
        # the plain workload: 10,000 mixture points, 1,000 components, 10 iterations, the default form
        {"name": "fit_fp64_10k_1k", "kind": "fit", "precision": "fp64", "N": 10000, "K": 1000, "iters": 10, "flags": 0},
        # a small scene in the default form (a first try, a unit test): launches and latency
        {"name": "fit_fp64_small", "kind": "fit", "precision": "fp64", "N": 1500, "K": 64, "iters": 4, "flags": 0},
        # the smallest ragged fit on the tensor cores: one point and one component past a tile
        {"name": "fit_fp16x3_ragged", "kind": "fit", "precision": "fp16x3", "N": 129, "K": 129, "iters": 3, "flags": 0},
        # the continual room stream of the benchmark: 200 x 200 frames, 50,000 components, 3 iterations per frame
        {"name": "stream_fp16x3_50k", "kind": "stream", "precision": "fp16x3", "side": 200, "K": 50000, "iters": 3,
         "flags": 0},
        # the same stream in the FP32 form (no tensor cores)
        {"name": "stream_fp32_50k", "kind": "stream", "precision": "fp32", "side": 200, "K": 50000, "iters": 3,
         "flags": 0},
        # the same model in the default FP64 form on 96 x 96 frames: a reference run of the stream
        {"name": "stream_fp64_50k", "kind": "stream", "precision": "fp64", "side": 96, "K": 50000, "iters": 3,
         "flags": 0},
        # a large map (200,000 components) with the learned proposal
        {"name": "stream_proposal_200k", "kind": "stream", "precision": "fp16x3", "side": 200, "K": 200000, "iters": 3,
         "flags": V.VBGS_FLAG_PROPOSAL},
        # scoring a frame under the map: compute_elbo_delta on its own
        {"name": "score_fp16x3_50k", "kind": "score", "precision": "fp16x3", "side": 200, "K": 50000, "flags": 0},
        # Alg. 1's step before fit: 1% of the components move to badly explained points
        {"name": "reassign_fp16x3_50k", "kind": "reassign", "precision": "fp16x3", "side": 200, "K": 50000, "n": 500,
         "flags": 0},
        # a view of the map
        {"name": "render_200", "kind": "render", "precision": "fp16x3", "side": 200, "K": 50000, "flags": 0},
        # eight uneven scenes in one call
        {"name": "batched_fp16x3_8", "kind": "batched", "precision": "fp16x3", "scenes": 8, "n_hi": 40000,
         "k_hi": 12000, "iters": 5, "flags": 0},
        # a host runtime that owns the device memory: odd sizes, the default form
        {"name": "estep_fp64_odd", "kind": "estep", "precision": "fp64", "N": 12345, "K": 1777, "flags": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "fit", "stream", "stream", "score", "reassign", "render", "batched", "estep"])
    precision = rng.choice(["fp64", "fp32", "fp16x3", "bf16x3"])
    split = V.VBGS_FLAG_SPLIT if rng.random() < 0.2 else 0
    if kind in ("fit", "estep"):
        N, K = _log_int(rng, 65, 20000), _log_int(rng, 17, 6000)
        c = {"kind": kind, "precision": precision, "N": N, "K": K, "flags": split}
        if kind == "fit":
            c["iters"] = rng.randint(1, 10)
        return c
    if kind == "batched":
        return {"kind": kind, "precision": rng.choice(["fp32", "fp16x3"]), "scenes": rng.randint(2, 12),
                "n_hi": _log_int(rng, 8000, 40000), "k_hi": _log_int(rng, 1500, 12000), "iters": rng.randint(1, 5),
                "flags": 0}
    if kind == "render":
        return {"kind": kind, "precision": "fp16x3", "side": _log_int(rng, 48, 400), "K": _log_int(rng, 2000, 50000),
                "flags": split}
    if precision == "bf16x3":     # 16-bit products do not hold the room's thin surfaces: not a form for a stream
        precision = "fp16x3"
    side = rng.randint(40, 96 if precision == "fp64" else 200)
    K = _log_int(rng, 1000, 50000)
    if kind == "stream":
        flags = split
        if precision != "fp64" and rng.random() < 0.2:
            flags |= V.VBGS_FLAG_PROPOSAL
        return {"kind": kind, "precision": precision, "side": side, "K": K, "iters": rng.randint(1, 3), "flags": flags}
    c = {"kind": kind, "precision": precision, "side": side, "K": K, "flags": split}
    if kind == "reassign":
        c["n"] = _log_int(rng, 16, 500)
    return c


# ---- inputs --------------------------------------------------------------------


def _points(case, seed):
    return synth.mixture_points(N=case["N"], seed=seed), synth.nw_prior(case["K"], seed + 100)


def _frames(case, seed):
    """Frames of a stream in order: those before the timed one, then those it
    cycles through (a render or a score needs only the first of them).  A
    sensor of a fixed number of returns: views that see at least 9 of 10 pixels
    within the depth range, thinned evenly to 9 of 10."""
    ahead = AHEAD if case["kind"] == "stream" else 1
    side = 200 if case["kind"] == "render" else case["side"]
    room, n, t, frames = synth.Room(seed), _returns(side), 0, []
    while len(frames) < WARM + ahead:
        f = synth.room_frame(t, seed=seed, width=side, height=side, room=room)
        t += 1
        if f.shape[0] >= n:
            frames.append(np.ascontiguousarray(f[np.arange(n) * f.shape[0] // n]))
    return frames[:WARM], frames[WARM:]


def _returns(side):
    return 9 * side * side // 10


def _scenes(case, seed):
    N, K = synth.scene_sizes(case["scenes"], seed=case["scenes"], n_lo=5000, n_hi=case["n_hi"], k_lo=1000,
                             k_hi=case["k_hi"])
    return [synth.c1_workload(seed + i, int(n), int(k)) for i, (n, k) in enumerate(zip(N, K))]


def _reassign_draws(case, seed, N):
    rng = np.random.default_rng([seed, 11])
    return rng.gumbel(size=N), rng.uniform(size=case["K"])


def _gpu(x):
    return torch.from_numpy(x).cuda()


def prepare(case, seed):
    kind, prec, flags = case["kind"], case["precision"], case["flags"]
    if kind == "batched":
        scenes = _scenes(case, seed)
        return {"case": case, "models": [V.Model(p, prec, flags=flags) for _, p in scenes],
                "points": [_gpu(x) for x, _ in scenes], "empty": [np.zeros((p["m0"].shape[0], F)) for _, p in scenes]}
    if kind in ("fit", "estep"):
        x, prior = _points(case, seed)
        m = V.Model(prior, prec, flags=flags)
        s = {"case": case, "model": m, "points": _gpu(x), "empty": np.zeros((case["K"], F))}
        if kind == "estep":
            m.update(s["points"], 2)
            s["lse"] = torch.empty(case["N"], dtype=torch.float64, device="cuda")
            s["stats"] = torch.empty((case["K"], F), dtype=torch.float64, device="cuda")
        return s
    warm, ahead = _frames(case, seed)
    m = V.Model(synth.room_prior(case["K"], seed=seed), prec, flags=flags)
    for f in warm:
        m.update(_gpu(f), case.get("iters", 3))
    s = {"case": case, "model": m, "frames": [_gpu(f) for f in ahead], "t": 0}
    if kind == "reassign":
        s["gumbel"], s["keys"] = _reassign_draws(case, seed, ahead[0].shape[0])
    if kind == "render":
        s["camera"] = synth.room_view(1000, seed=seed, width=case["side"], height=case["side"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "fit":
        m = s["model"]
        m.set_stats(s["empty"])
        return {"elbo": m.update(s["points"], case["iters"]), "stats": m.stats()}
    if kind == "stream":
        m, f = s["model"], s["frames"][s["t"] % len(s["frames"])]
        s["t"] += 1
        return {"elbo": m.update(f, case["iters"]), "stats": m.frame_stats()}
    if kind == "score":
        elbo, lse = s["model"].elbo(s["frames"][0], want_lse=True)
        return {"elbo": elbo, "lse": lse}
    if kind == "reassign":
        m, f = s["model"], s["frames"][0]
        points, comps = m.reassign(f, case["n"], s["gumbel"], 1.0, s["keys"])
        return {"points": points, "components": comps, "lse": m.lse(f.shape[0])}
    if kind == "render":
        return s["model"].render(s["camera"])[0]
    if kind == "batched":
        for m, z in zip(s["models"], s["empty"]):
            m.set_stats(z)
        traces = V.vbgs_update_batched([m.ctx for m in s["models"]], s["points"], case["iters"])
        return {"elbo": traces, "stats": [m.stats() for m in s["models"]]}
    V.vbgs_estep_noalloc(s["model"].ctx, s["points"], s["lse"], s["stats"], case["K"])
    return {"lse": s["lse"], "stats": s["stats"]}


def work(case):
    """Bytes: points in (N x 6 doubles), statistics in and out (K x 28
    doubles), per-point terms or pixels out.  Flops: the two contractions of
    the update as the method states them (28 features, 56 flops per point and
    component each); the library leaves out pairs it certifies negligible."""
    kind = case["kind"]
    if kind == "batched":
        N, K = synth.scene_sizes(case["scenes"], seed=case["scenes"], n_lo=5000, n_hi=case["n_hi"], k_lo=1000,
                                 k_hi=case["k_hi"])
        pairs = float(np.sum(N.astype(float) * K)) * case["iters"]
        return {"bytes": float(48 * N.sum() + 2 * 224 * K.sum()), "flops": 112.0 * pairs}
    K = float(case["K"])
    if kind == "render":
        return {"bytes": 224.0 * K + 12.0 * case["side"] ** 2, "flops": 0.0}
    N = float(case["N"]) if "N" in case else float(_returns(case["side"]))
    if kind in ("score", "reassign"):
        return {"bytes": 56.0 * N + 224.0 * K, "flops": 56.0 * N * K}
    iters = case.get("iters", 1)
    return {"bytes": 48.0 * N + 2 * 224.0 * K, "flops": 112.0 * N * K * iters}


# ---- the update in 64 bits -----------------------------------------------------


class _Exact:
    """Mean-field Normal-Wishart / Dirichlet mixture, raw-moment statistics."""

    def __init__(self, prior, split):
        f8 = {"dtype": torch.float64, "device": "cuda"}
        self.a0, self.b0, self.n0 = prior["alpha0"], prior["beta0"], prior["nu0"]
        self.m0 = torch.as_tensor(prior["m0"], **f8)
        self.K = self.m0.shape[0]
        self.blocks = [(0, 3), (3, 6)] if split else [(0, 6)]
        self.W0i = torch.zeros((D, D), **f8)
        W0 = torch.as_tensor(prior["W0"], **f8)
        for lo, hi in self.blocks:
            self.W0i[lo:hi, lo:hi] = torch.linalg.inv(W0[lo:hi, lo:hi])
        self.iu = torch.triu_indices(D, D, device="cuda")

    def posterior(self, S):
        n = S[:, 0]
        alpha, beta, nu = self.a0 + n, self.b0 + n, self.n0 + n
        m = (self.b0 * self.m0 + S[:, 1:7]) / beta[:, None]
        S2 = torch.zeros((self.K, D, D), dtype=torch.float64, device="cuda")
        S2[:, self.iu[0], self.iu[1]] = S[:, 7:]
        S2[:, self.iu[1], self.iu[0]] = S[:, 7:]
        outer = lambda v: v[:, :, None] * v[:, None, :]  # noqa: E731
        A = self.W0i + S2 + self.b0 * outer(self.m0) - beta[:, None, None] * outer(m)
        if len(self.blocks) == 2:
            A[:, :3, 3:] = 0
            A[:, 3:, :3] = 0
        L = torch.linalg.cholesky(A)
        return {"alpha": alpha, "beta": beta, "nu": nu, "m": m, "L": L}

    def _mv(self, f, a, d):
        return sum(f(a - 0.5 * i) for i in range(d))

    def records(self, q):
        """c_k and M_k of log rho_nk = c_k - |M_k (x - m_k)|^2 / 2."""
        ld = 2 * torch.log(torch.diagonal(q["L"], dim1=1, dim2=2)).sum(1)
        psi = sum(self._mv(torch.special.digamma, 0.5 * q["nu"], hi - lo) for lo, hi in self.blocks)
        c = (torch.special.digamma(q["alpha"]) - torch.special.digamma(q["alpha"].sum())
             + 0.5 * (psi + D * math.log(2) - ld) - 0.5 * D * math.log(2 * math.pi) - 0.5 * D / q["beta"])
        eye = torch.eye(D, dtype=torch.float64, device="cuda").expand(self.K, D, D)
        M = torch.linalg.solve_triangular(q["L"], eye, upper=False) * torch.sqrt(q["nu"])[:, None, None]
        return c, M

    def estep(self, q, X, stats=True):
        c, M = self.records(q)
        Mm = torch.einsum("kij,kj->ki", M, q["m"]).reshape(-1)
        Mt = M.reshape(self.K * D, D).T.contiguous()
        lse, S = [], torch.zeros((self.K, F), dtype=torch.float64, device="cuda")
        step = max(1, int(4e8) // (self.K * D))
        for i in range(0, X.shape[0], step):
            x = X[i:i + step]
            y = torch.addmm(-Mm, x, Mt).square_().view(-1, self.K, D)
            l = y.sum(2).mul_(-0.5).add_(c)
            z = torch.logsumexp(l, 1)
            lse.append(z)
            if stats:
                phi = torch.cat([torch.ones_like(x[:, :1]), x, x[:, self.iu[0]] * x[:, self.iu[1]]], 1)
                S += torch.exp(l.sub_(z[:, None])).T @ phi
        return (torch.cat(lse) if lse else torch.zeros(0, dtype=torch.float64, device="cuda")), S

    def kl(self, q, p):
        tot = torch.zeros(self.K, dtype=torch.float64, device="cuda")
        lg = torch.special.gammaln
        for lo, hi in self.blocks:
            d = hi - lo
            Lq, Lp = q["L"][:, lo:hi, lo:hi], p["L"][:, lo:hi, lo:hi]
            dm = (q["m"] - p["m"])[:, lo:hi]
            w = torch.linalg.solve_triangular(Lq, dm[:, :, None], upper=False)[:, :, 0].square().sum(1)
            tr = torch.linalg.solve_triangular(Lq, Lp, upper=False).square().sum((1, 2))
            ld = lambda L: 2 * torch.log(torch.diagonal(L, dim1=1, dim2=2)).sum(1)  # noqa: E731
            bq, bp, nq, np_ = q["beta"], p["beta"], q["nu"], p["nu"]
            tot += 0.5 * (d * (bp / bq - 1 + torch.log(bq / bp)) + bp * nq * w)
            tot += 0.5 * np_ * (ld(Lq) - ld(Lp)) + 0.5 * nq * (tr - d)
            tot += self._mv(lg, 0.5 * np_, d) - self._mv(lg, 0.5 * nq, d)
            tot += 0.5 * (nq - np_) * self._mv(torch.special.digamma, 0.5 * nq, d)
        a, b = q["alpha"], p["alpha"]
        dirichlet = (lg(a.sum()) - lg(b.sum()) + (lg(b) - lg(a)
                     + (a - b) * (torch.special.digamma(a) - torch.special.digamma(a.sum()))).sum())
        return tot.sum() + dirichlet

    def frame(self, S, X, iters):
        p = q = self.posterior(S)
        trace, dS = [], None
        for i in range(iters):
            lse, dS = self.estep(q, X)
            trace.append(float(lse.sum() - (self.kl(q, p) if i else 0.0)))
            q = self.posterior(S + dS)
        return np.array(trace), dS


def exact(case, seed):
    kind = case["kind"]
    split = bool(case["flags"] & V.VBGS_FLAG_SPLIT)
    frames = WARM + 1
    if kind == "render" or (kind == "stream" and _returns(case["side"]) * case["K"] * case["iters"] * frames > 3e10):
        return None
    empty = lambda K: torch.zeros((K, F), dtype=torch.float64, device="cuda")  # noqa: E731
    if kind == "batched":
        out = []
        for x, prior in _scenes(case, seed):
            e = _Exact(prior, split)
            out.append(e.frame(empty(e.K), _gpu(x), case["iters"]))
        return {"elbo": np.stack([t for t, _ in out]), "stats": [s.cpu().numpy() for _, s in out]}
    if kind in ("fit", "estep"):
        x, prior = _points(case, seed)
        e, x = _Exact(prior, split), _gpu(x)
        trace, S = e.frame(empty(e.K), x, case.get("iters", 2))
        if kind == "fit":
            return {"elbo": trace, "stats": S.cpu().numpy()}
        lse, dS = e.estep(e.posterior(S), x)
        return {"lse": lse, "stats": dS}
    warm, ahead = _frames(case, seed)
    e = _Exact(synth.room_prior(case["K"], seed=seed), split)
    S = empty(e.K)
    for f in warm:
        S = S + e.frame(S, _gpu(f), case.get("iters", 3))[1]
    x = _gpu(ahead[0])
    if kind == "stream":
        trace, dS = e.frame(S, x, case["iters"])
        return {"elbo": trace, "stats": dS.cpu().numpy()}
    lse = e.estep(e.posterior(S), x, stats=False)[0].cpu().numpy()
    if kind == "score":
        return {"elbo": float(lse.sum()), "lse": lse}
    return {"points": None, "components": None, "lse": lse}
