"""The calls whose time counts: what a user of this library has it do.

Every case is one call of a public entry point on an ensemble of noise
realizations, at sizes of the named workloads (shortened in steps, and where
the run would take long in realizations) or of the paper's own benchmark: a
ring with noisy couplings, 1000 realizations, N^2 between 10^3 and 10^4.
draw() spreads the same families over their ranges: lattice sizes 16..4096
(odd ones among them), 1..2048 realizations, orders 4..20, rings and open
chains, the three statistics, both state types, with and without samples.

A pass starts from a spread-out, normalised state in device memory (what a
run meets most of its time; a walker starts on one site and spreads) and
returns the final states and the sampled observables.  The observables of
complex64 runs are FP64 sums over FP32 amplitudes; they are handed on in the
state's precision, as a program that plots or fits them would.
"""
import math

import numpy as np
import torch

from paper_1612_00746_gb300 import ctqw

DIST, BOSONS, FERMIONS = ctqw.DISTINGUISHABLE, ctqw.BOSONS, ctqw.FERMIONS


def _chain(name, **kw):
    c = dict(name=name, kind="taylor", m=2, stats=DIST, ring=False, N=64, N_max=0, N_step=0, R=1, U=0.0, eps=1.0,
             J=0.0, dt=0.02, K=16, steps=10, every=0, fp64=False)
    c.update(kw)
    return c


def listed():
    return [
        # One trajectory advanced a little, as an interactive program or the
        # inner loop of a fit does: launches and latency.
        _chain("one_n64", stats=BOSONS, N=64, R=1, U=2.0, J=0.25, steps=10),
        # The plain FP64 method on a handful of realizations, sampled every
        # 10 steps (fp64_plain_n64, a fifth of its steps).
        _chain("fp64_n64", N=64, R=8, eps=0.5, dt=0.01, K=12, steps=200, every=10, fp64=True),
        # The headline: bosons_n256_u2 with all of its realizations.
        _chain("bosons_n256", stats=BOSONS, N=256, R=1024, U=2.0, J=0.25, steps=50, every=10),
        # The paper's own benchmark: a ring, noise on the couplings, 1000
        # realizations, 10^4 amplitudes each, post-processed now and then.
        _chain("ring_n100", ring=True, N=100, R=1000, eps=0.0, J=0.25, steps=100, every=25),
        # A batch of uneven sizes (ragged_n128_1024, a quarter of it).
        _chain("ragged_n128_1024", N=128, N_max=1024, N_step=64, R=512, U=1.0, J=0.25, K=8, steps=20, every=10),
        # One gradient of a fit to a target occupation (adjoint_n512).
        _chain("adjoint_n512", kind="adjoint", N=512, R=64, eps=0.2, J=0.2, K=14, steps=50, every=25),
        # Three bosons on a ring (ring3_n160).
        _chain("ring3_n160", m=3, stats=BOSONS, ring=True, N=160, R=16, U=2.0, dt=0.01, steps=10, every=5),
        # Large FP64 states (dist_n4096_c128).
        _chain("fp64_n4096", N=4096, R=4, U=2.0, dt=0.01, steps=5, fp64=True),
        # Two bosons on the 15 x 15 torus (lattice2d_15x15_m2).
        _chain("lattice_15x15", kind="graph", stats=BOSONS, ring=True, N=15, N_max=15, R=1000, U=2.0, J=0.25, steps=20,
               every=10),
        # The ensemble's one-body density matrix of the headline states.
        _chain("density_n256", kind="density", stats=BOSONS, N=256, R=1024, U=2.0, J=0.25),
        # Switching noise, the paper's own kind: H changes after every step.
        _chain("switching_n256", kind="switching", stats=BOSONS, N=256, R=256, U=2.0, J=0.25, steps=50, every=10),
        # The paper's second propagator, in FP64, where its comparison of
        # the two methods is made.
        _chain("rk4_fp64_n256", kind="rk4", stats=BOSONS, N=256, R=16, U=2.0, J=0.25, K=4, steps=100, every=10,
               fp64=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# Site-updates of the listed case of each family, which drawn ones stay
# within: two particles in FP32, in FP64, three particles, graphs.
_CAP = {"taylor": 5.0e10, "taylor64": 5.0e9, "taylor3": 1.0e10, "switching": 1.3e10, "rk4": 4.0e8, "rk432": 1.5e10,
        "adjoint": 1.1e10, "graph": 1.6e10, "density": 6.8e7}


def draw(rng):
    kind = rng.choice(["taylor", "taylor", "taylor", "ragged", "taylor64", "taylor64", "taylor3", "switching", "rk4",
                       "rk432", "adjoint", "graph", "density"])
    ring, stats = rng.random() < 0.4, rng.choice([DIST, BOSONS, FERMIONS])
    every = rng.choice([0, 5, 10, 25])
    c = dict(kind=kind, m=2, stats=stats, ring=ring, N=0, N_max=0, N_step=0, R=_log_int(rng, 1, 2048),
             U=rng.choice([0.0, 1.0, 2.0]), eps=rng.choice([0.0, 0.5, 1.0]), J=rng.choice([0.0, 0.25]),
             dt=rng.choice([0.01, 0.02]), K=rng.randint(6, 20), steps=_log_int(rng, 4, 100), every=every, fp64=False)
    if kind == "graph":
        c["N"] = rng.randint(3, 16)
        c["N_max"] = rng.randint(3, 16)
        c["R"] = _log_int(rng, 1, 1500)
        c["fp64"] = rng.random() < 0.25
    elif kind == "ragged":
        c["kind"] = "taylor"
        c["N_step"] = rng.choice([1, 32, 64])
        c["N"] = rng.choice([64, 128, 192])
        c["N_max"] = c["N"] + 64 * rng.randint(1, 13)
        c["K"] = rng.randint(6, 16)
    elif kind == "taylor3":
        c["kind"], c["m"] = "taylor", 3
        c["N"] = _log_int(rng, 12, 160)
        c["fp64"] = rng.random() < 0.25
    elif kind in ("taylor64", "rk4"):
        c["kind"] = "taylor" if kind == "taylor64" else "rk4"
        c["N"] = _log_int(rng, 16, 4096 if kind == "taylor64" else 256)
        c["fp64"] = True
    elif kind == "rk432":
        c["kind"] = "rk4"
        c["N"] = rng.choice([64, 128, 192, 256, _log_int(rng, 16, 512)])
    elif kind == "adjoint":
        c["N"] = _log_int(rng, 32, 512)
        c["every"] = rng.choice([5, 10, 25, 50])
        c["fp64"] = rng.random() < 0.25
        c["R"] = _log_int(rng, 1, 256)
    elif kind == "density":
        c["N"] = _log_int(rng, 16, 1024)
        c["fp64"] = rng.random() < 0.25
        c["steps"], c["every"] = 0, 0
    else:
        c["N"] = rng.choice([64, 128, 192, 256, _log_int(rng, 16, 1024), _log_int(rng, 16, 1024)])
    if c["kind"] == "rk4":
        c["K"] = 4
    # within the family's share of work: fewer realizations, then fewer steps
    cap = _CAP[{"ragged": "taylor"}.get(kind, kind)]
    if kind in ("taylor3", "adjoint", "graph", "density") and c["fp64"]:
        cap /= 12.0
    sites = _mean_states(c)
    per = sites * (1 if kind == "density" else c["K"] * c["steps"])
    c["R"] = max(1, min(c["R"], int(cap / per)))
    if kind != "density":
        c["steps"] = max(1, min(c["steps"], int(cap / (sites * c["K"] * c["R"]))))
    if kind == "adjoint":
        c["every"] = max(1, min(c["every"], c["steps"]))
    elif c["every"] > c["steps"]:
        c["every"] = c["steps"]
    return c


def _nodes(c):
    return c["N"] * c["N_max"] if c["kind"] == "graph" else c["N"]


def _mean_states(c):
    """Amplitudes of a realization (the mean over the range of a ragged batch)."""
    if c["N_step"]:
        n = np.arange(c["N"], c["N_max"] + 1, c["N_step"], dtype=np.float64)
        return float(np.mean(n ** c["m"]))
    return float(_nodes(c)) ** c["m"]


def _sizes(c):
    if c["N_step"]:
        # the sizes of the batch are part of the workload, not of its noise
        g = np.random.Generator(np.random.PCG64(c["R"]))
        return g.choice(np.arange(c["N"], c["N_max"] + 1, c["N_step"]), size=c["R"]).astype(np.int64)
    return np.full(c["R"], c["N"], dtype=np.int64)


def _edges(c):
    """Links of the N x N_max lattice, periodic when the case is a ring."""
    idx = np.arange(c["N"] * c["N_max"]).reshape(c["N"], c["N_max"])
    us, vs = [], []
    for axis, n in enumerate(idx.shape):
        nxt, src = np.roll(idx, -1, axis=axis), idx
        if not c["ring"]:
            keep = (slice(0, n - 1), slice(None)) if axis == 0 else (slice(None), slice(0, n - 1))
            src, nxt = idx[keep], nxt[keep]
        us.append(src.reshape(-1))
        vs.append(nxt.reshape(-1))
    return np.concatenate(us).astype(np.int32), np.concatenate(vs).astype(np.int32)


def _draws(c, seed):
    """Uniform draws of the disorder (eps, J), packed over the realizations."""
    g = np.random.Generator(np.random.Philox(np.random.SeedSequence([int(seed), 17])))
    if c["kind"] == "graph":
        n, e = _nodes(c), len(_edges(c)[0])
        return g.random((c["R"], n)), g.random((c["R"], e))
    n = int(_sizes(c).sum())
    return g.random(n), g.random(n)


def _envelope(n, gen):
    x = torch.arange(n, device="cuda", dtype=torch.float32)
    centre = n * (0.4 + 0.2 * torch.rand(1, generator=gen, device="cuda"))
    return torch.exp(-((x - centre) / (0.3 * n)) ** 2)


def _states(c, n, count, gen):
    """`count` normalised states of n^m amplitudes: random phases under an
    envelope, (anti)symmetrised like the statistics; complex64 values."""
    m = c["m"]
    out = torch.view_as_complex(torch.randn((count,) + (n,) * m + (2,), generator=gen, device="cuda"))
    env = _envelope(n, gen)
    for a in range(1, m + 1):
        out *= env.view((-1,) + (1,) * (m - a))
    if c["stats"] != DIST:
        sign = 1.0 if c["stats"] == BOSONS else -1.0
        if m == 2:
            out = out + sign * out.transpose(1, 2)
        else:
            out = out + sign * out.transpose(1, 2)
            out = out + out.permute(0, 3, 1, 2) + out.permute(0, 2, 3, 1)
    out /= torch.linalg.vector_norm(out.reshape(count, -1), dim=1).clamp_min(1e-20).view((-1,) + (1,) * m)
    return out.contiguous()


def _psi0(c, seed):
    """The initial states in the library's layout, and (torch) complex64 or complex128."""
    gen = torch.Generator("cuda")
    gen.manual_seed(int(seed))
    dtype = torch.complex128 if c["fp64"] else torch.complex64
    if c["kind"] == "graph":
        n, R = _nodes(c), c["R"]
        Rp = (R + 3) // 4 * 4
        psi = torch.zeros(n * n, Rp, dtype=dtype, device="cuda")
        psi[:, :R] = _states(c, n, R, gen).reshape(R, -1).t()
        return psi.reshape(-1)
    sizes = _sizes(c)
    if not c["N_step"]:
        return _states(c, c["N"], c["R"], gen).reshape(-1).to(dtype)
    return torch.cat([_states(c, int(n), 1, gen).reshape(-1).to(dtype) for n in sizes])


def _target(c, width, seed):
    gen = torch.Generator("cuda")
    gen.manual_seed(int(seed) + 99)
    t = torch.rand(width, generator=gen, device="cuda", dtype=torch.float64) + 0.1
    return t / t.sum()


_SWITCH_P = 0.01


def prepare(case, seed):
    c = case
    dtype = ctqw.C128 if c["fp64"] else ctqw.C64
    ue, uj = _draws(c, seed)
    s = {"case": c, "dtype": dtype, "seed": int(seed)}
    if c["kind"] == "graph":
        u, v = _edges(c)
        h = ctqw.Graph(2, c["stats"], _nodes(c), u, v, c["R"], 1.0, c["U"], c["eps"], c["J"], ue, uj)
        s["ws"] = h.workspace(dtype)
        width = h.N
    else:
        h = ctqw.Hamiltonian(c["m"], c["stats"], c["ring"], _sizes(c), 1.0, c["U"], c["eps"], c["J"], ue, uj)
        width = h.p_width
        if c["kind"] == "adjoint":
            s["target"] = _target(c, width, seed)
            s["ws"] = ctqw.adjoint_workspace(h, dtype, c["K"], c["steps"], c["every"])
        elif c["kind"] == "switching":
            s["ws"] = h.workspace(dtype, ctqw.TAYLOR, ctqw.FLAG_PLAIN)
        elif c["kind"] != "density":
            s["ws"] = h.workspace(dtype, ctqw.RK4 if c["kind"] == "rk4" else ctqw.TAYLOR)
    s["h"] = h
    s["psi0"] = _psi0(c, seed)
    s["psi"] = torch.empty_like(s["psi0"])
    n_obs = c["steps"] // c["every"] + 1 if c["every"] and c["kind"] not in ("adjoint", "density") else 0
    f64 = dict(dtype=torch.float64, device="cuda")
    s["P"] = torch.empty((n_obs, width), **f64) if n_obs else None
    s["norm"] = torch.empty((n_obs, h.R), **f64) if n_obs else None
    s["energy"] = torch.empty((n_obs, h.R), **f64) if n_obs else None
    return s


def _handed_on(state, values):
    """FP64 outputs in the precision of the states they were formed from."""
    if state["dtype"] == ctqw.C128:
        return values
    low = {torch.float64: torch.float32, torch.complex128: torch.complex64}
    return {k: (v.to(low.get(v.dtype, v.dtype)) if v is not None else None) for k, v in values.items()}


def run(state):
    c, h, dtype, psi = state["case"], state["h"], state["dtype"], state["psi"]
    P, norm, energy = state["P"], state["norm"], state["energy"]
    if c["kind"] == "density":
        rho = ctqw.ctqw_one_body_density(h, state["psi0"], dtype)
        return _handed_on(state, {"rho": rho[0]})
    if c["kind"] == "adjoint":
        loss, ge, gJ, Pf, gem, gJm = ctqw.ctqw_adjoint_grad(h, state["psi0"], dtype, c["dt"], c["K"], c["steps"],
                                                            c["every"], state["target"], workspace=state["ws"])
        return _handed_on(state, {"loss": loss, "grad_eps": ge, "grad_J": gJ, "P": Pf, "grad_eps_mean": gem,
                                  "grad_J_mean": gJm})
    psi.copy_(state["psi0"])
    if c["kind"] == "graph":
        ctqw.ctqw_graph_propagate_taylor(h, psi, dtype, c["dt"], c["K"], c["steps"], c["every"], P, norm, energy,
                                         state["ws"])
    elif c["kind"] == "switching":
        ctqw.ctqw_propagate_taylor_switching(h, psi, dtype, c["dt"], c["K"], c["steps"], c["every"], P, norm, energy,
                                             state["seed"], _SWITCH_P, workspace=state["ws"])
    elif c["kind"] == "rk4":
        ctqw.ctqw_propagate_rk4(h, psi, dtype, c["dt"], c["steps"], c["every"], P, norm, energy,
                                workspace=state["ws"])
    else:
        ctqw.ctqw_propagate_taylor(h, psi, dtype, c["dt"], c["K"], c["steps"], c["every"], P, norm, energy,
                                   workspace=state["ws"])
    out = _handed_on(state, {"P": P, "norm": norm, "energy": energy})
    out["psi"] = psi
    return out


def work(case):
    """Each state read and written once a call, the outputs written once; the
    products and sums of the stencil: (8m + 4) flops per amplitude and term
    (a graph: 4 per link end and particle, and 8)."""
    c = case
    b = 16 if c["fp64"] else 8
    sites = float(np.sum(_sizes(c).astype(np.float64) ** c["m"])) if c["kind"] != "graph" else \
        c["R"] * float(_nodes(c)) ** 2
    width = _nodes(c) if not c["N_step"] else int(np.unique(_sizes(c)).sum())
    if c["kind"] == "density":
        return {"bytes": sites * b + 16.0 * width * width, "flops": 8.0 * c["m"] * sites * c["N"]}
    n_obs = c["steps"] // c["every"] + 1 if c["every"] and c["kind"] != "adjoint" else 0
    out = 8.0 * n_obs * (width + 2 * c["R"])
    terms = sites * c["K"] * c["steps"]
    if c["kind"] == "graph":
        per = 8.0 + 4.0 * c["m"] * 2.0 * len(_edges(c)[0]) / _nodes(c)
        return {"bytes": 2 * b * sites + out, "flops": per * terms}
    params = 16.0 * float(_sizes(c).sum())
    if c["kind"] == "adjoint":
        # forward terms, the reverse recurrence and the gradient's products
        return {"bytes": b * sites + 2 * params + 24.0 * width, "flops": 3.0 * (8 * c["m"] + 4) * terms}
    return {"bytes": 2 * b * sites + params + out, "flops": (8.0 * c["m"] + 4.0) * terms}


# ------------------------------------------------------------ values in FP64
# States as real tensors [count, n, .., n, 2] (re, im); H is real.

def _round(v):
    return np.asarray(v, dtype=np.float64).astype(np.float32).astype(np.float64)


def _params(c, seed):
    """Per realization (eps [n], J [n]) as FP64 arrays of float32 values."""
    ue, uj = _draws(c, seed)
    off = np.concatenate([[0], np.cumsum(_sizes(c))])
    eps, J = _round(c["eps"] * (2.0 * ue - 1.0)), _round(1.0 + c["J"] * (2.0 * uj - 1.0))
    out = []
    for r in range(c["R"]):
        e, j = eps[off[r]:off[r + 1]], J[off[r]:off[r + 1]].copy()
        if not c["ring"]:
            j[-1] = 0.0
        out.append((e, j))
    return out


def _pairs(n, m):
    x = torch.arange(n, device="cuda")
    if m == 2:
        return (x.view(-1, 1) == x).double()
    a, b, d = x.view(-1, 1, 1), x.view(1, -1, 1), x.view(1, 1, -1)
    return (a == b).double() + (a == d).double() + (b == d).double()


def _along(v, axis, m):
    """[count, n] values along one coordinate of [count, n, .., n, 2]."""
    shape = [v.shape[0]] + [1] * m + [1]
    shape[1 + axis] = v.shape[1]
    return v.view(shape)


def _apply(psi, eps, J, U, pairs, m):
    v = _along(eps, 0, m)
    for a in range(1, m):
        v = v + _along(eps, a, m)
    if U:
        v = v + (U * pairs).unsqueeze(0).unsqueeze(-1)
    y = v * psi
    Jl = torch.roll(J, 1, 1)
    for a in range(m):
        y = y - _along(Jl, a, m) * torch.roll(psi, 1, 1 + a)
        y = y - _along(J, a, m) * torch.roll(psi, -1, 1 + a)
    return y


def _times(y, k):
    """-i k y."""
    return torch.stack((k * y[..., 1], -k * y[..., 0]), -1)


def _step(psi, apply, dt, K):
    phi, acc = psi, psi
    for j in range(1, K + 1):
        phi = _times(apply(phi), dt / j)
        acc = acc + phi
    return acc


def _observe(psi, apply, m):
    """(P summed over the realizations, norm, energy) of a block of states."""
    p = psi.square().sum(-1)
    dims = tuple(range(1, m + 1))
    P = sum(p.sum(tuple(d for d in dims if d != a)).sum(0) for a in dims) / m
    return P, p.sum(dims), (psi * apply(psi)).sum(dims + (m + 1,))


def _switched(c, seed, step, eps, J):
    """The parameters after the update that follows `step` (Philox4x64-10)."""
    R, n = eps.shape
    u32 = np.uint64(0xFFFFFFFF)

    def product(a, b):   # 64 x 64 -> (high, low)
        a0, a1, b0, b1 = a & u32, a >> np.uint64(32), b & u32, b >> np.uint64(32)
        t = a1 * b0 + ((a0 * b0) >> np.uint64(32))
        w = (t & u32) + a0 * b1
        return a1 * b1 + (t >> np.uint64(32)) + (w >> np.uint64(32)), a * b

    with np.errstate(over="ignore"):
        w = [np.full((R, n), step, np.uint64), np.repeat(np.arange(R, dtype=np.uint64)[:, None], n, 1),
             np.repeat(np.arange(n, dtype=np.uint64)[None], R, 0), np.zeros((R, n), np.uint64)]
        k0, k1 = np.uint64(seed), np.uint64(0)
        for _ in range(10):
            h0, l0 = product(np.uint64(0xD2E7470EE14C6C93), w[0])
            h1, l1 = product(np.uint64(0xCA5A826395121157), w[2])
            w = [h1 ^ w[1] ^ k0, l1, h0 ^ w[3] ^ k1, l0]
            k0, k1 = k0 + np.uint64(0x9E3779B97F4A7C15), k1 + np.uint64(0xBB67AE8584CAA73B)
    u = [(x >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 for x in w]
    eps = np.where(u[0] < _SWITCH_P, _round(c["eps"] * (2.0 * u[1] - 1.0)), eps)
    Jn = np.where(u[2] < _SWITCH_P, _round(1.0 + c["J"] * (2.0 * u[3] - 1.0)), J)
    if not c["ring"]:
        Jn[:, -1] = 0.0
    return eps, Jn


def _exact_chain(c, seed):
    m, K = c["m"], c["K"]
    sizes, params = _sizes(c), _params(c, seed)
    psi0 = torch.view_as_real(_psi0(c, seed))
    off = np.concatenate([[0], np.cumsum(sizes ** m)])
    groups = np.unique(sizes)
    n_obs = c["steps"] // c["every"] + 1 if c["every"] else 0
    P = torch.zeros(n_obs, int(groups.sum()), dtype=torch.float64, device="cuda")
    norm = torch.zeros(n_obs, c["R"], dtype=torch.float64, device="cuda")
    energy = torch.zeros_like(norm)
    final = torch.empty(int(off[-1]), 2, dtype=torch.float64, device="cuda")
    at = 0
    for n in groups:
        n = int(n)
        members = np.flatnonzero(sizes == n)
        pairs = _pairs(n, m)
        block = len(members) if c["kind"] == "switching" else max(1, int(2e8 / n ** m))
        for b in range(0, len(members), block):
            ids = members[b:b + block]
            rs = torch.from_numpy(ids).cuda()
            eps_h, J_h = np.stack([params[r][0] for r in ids]), np.stack([params[r][1] for r in ids])
            eps, J = torch.from_numpy(eps_h).cuda(), torch.from_numpy(J_h).cuda()
            psi = torch.stack([psi0[off[r]:off[r + 1]] for r in ids]).double().view((len(ids),) + (n,) * m + (2,))

            def apply(x):
                return _apply(x, eps, J, c["U"], pairs, m)

            for step in range(c["steps"] + 1):
                if n_obs and step % c["every"] == 0:
                    p, nr, en = _observe(psi, apply, m)
                    q = step // c["every"]
                    P[q, at:at + n] += p / len(members)
                    norm[q, rs], energy[q, rs] = nr, en
                if step == c["steps"]:
                    break
                psi = _step(psi, apply, c["dt"], K)
                if c["kind"] == "switching":
                    eps_h, J_h = _switched(c, seed, step, eps_h, J_h)
                    eps, J = torch.from_numpy(eps_h).cuda(), torch.from_numpy(J_h).cuda()
            for k, r in enumerate(ids):
                final[off[r]:off[r + 1]] = psi[k].reshape(-1, 2)
        at += n
    out = {"P": P, "norm": norm, "energy": energy} if n_obs else {"P": None, "norm": None, "energy": None}
    out["psi"] = torch.view_as_complex(final)
    return out


def _exact_graph(c, seed):
    n, R = _nodes(c), c["R"]
    Rp = (R + 3) // 4 * 4
    ue, uj = _draws(c, seed)
    u, v = (torch.from_numpy(x.astype(np.int64)).cuda() for x in _edges(c))
    eps = torch.zeros(n, Rp, dtype=torch.float64, device="cuda")
    J = torch.zeros(len(u), Rp, dtype=torch.float64, device="cuda")
    eps[:, :R] = torch.from_numpy(_round(c["eps"] * (2.0 * ue - 1.0))).cuda().t()
    J[:, :R] = torch.from_numpy(_round(1.0 + c["J"] * (2.0 * uj - 1.0))).cuda().t()
    V = (eps.view(n, 1, Rp) + eps.view(1, n, Rp) + c["U"] * _pairs(n, 2).unsqueeze(-1)).unsqueeze(-1)
    # every node's links, padded with links of no weight
    ends = [[] for _ in range(n)]
    for e, (a, b) in enumerate(zip(u.tolist(), v.tolist())):
        ends[a].append((b, e))
        ends[b].append((a, e))
    J = torch.cat([J, torch.zeros(1, Rp, dtype=torch.float64, device="cuda")])
    tables = []
    for k in range(max(len(x) for x in ends)):
        pick = [x[k] if k < len(x) else (0, len(u)) for x in ends]
        tables.append((torch.tensor([p[0] for p in pick], device="cuda"), torch.tensor([p[1] for p in pick], device="cuda")))

    def apply(x):
        y = V * x
        for node, link in tables:
            w = J[link].unsqueeze(-1)
            y -= w.unsqueeze(1) * x[node]
            y -= w.unsqueeze(0) * x[:, node]
        return y

    psi = torch.view_as_real(_psi0(c, seed)).double().view(n, n, Rp, 2)
    P, norm, energy = [], [], []
    for step in range(c["steps"] + 1):
        if c["every"] and step % c["every"] == 0:
            p = psi.square().sum(-1)[..., :R]
            P.append((p.sum((1, 2)) + p.sum((0, 2))) / (2.0 * R))
            norm.append(p.sum((0, 1)))
            energy.append((psi * apply(psi)).sum((0, 1, 3))[:R])
        if step == c["steps"]:
            break
        psi = _step(psi, apply, c["dt"], c["K"])
    out = {"P": torch.stack(P), "norm": torch.stack(norm), "energy": torch.stack(energy)} if P else \
        {"P": None, "norm": None, "energy": None}
    out["psi"] = torch.view_as_complex(psi.contiguous()).reshape(-1)
    return out


def _exact_adjoint(c, seed):
    n, R, K = c["N"], c["R"], c["K"]
    params = _params(c, seed)
    eps = torch.from_numpy(np.stack([p[0] for p in params])).cuda()
    J = torch.from_numpy(np.stack([p[1] for p in params])).cuda()
    pairs = _pairs(n, 2)
    target = _target(c, n, seed)
    trail = [torch.view_as_real(_psi0(c, seed)).double().view(R, n, n, 2)]

    def step(x, e, j):
        return _step(x, lambda z: _apply(z, e, j, c["U"], pairs, 2), c["dt"], K)

    for _ in range(c["steps"]):
        trail.append(step(trail[-1], eps, J))
    p = trail[-1].square().sum(-1)
    P = (p.sum((0, 2)) + p.sum((0, 1))) / (2.0 * R)
    loss = (P - target).square().sum()
    g = (P - target) * 2.0 / (2.0 * R)   # d loss / d p_r(x1, x2) = g(x1) + g(x2)
    lam = 2.0 * (g.view(1, n, 1, 1) + g.view(1, 1, n, 1)) * trail[-1]
    ge, gJ = torch.zeros_like(eps), torch.zeros_like(J)
    for k in range(c["steps"] - 1, -1, -1):
        e, j = eps.clone().requires_grad_(), J.clone().requires_grad_()
        x = trail[k].clone().requires_grad_()
        with torch.enable_grad():
            y = step(x, e, j)
        lam, de, dj = torch.autograd.grad(y, (x, e, j), lam)
        ge += de
        gJ += dj
    if not c["ring"]:
        gJ[:, -1] = 0.0
    return {"loss": loss.reshape(1), "grad_eps": ge.reshape(-1), "grad_J": gJ.reshape(-1), "P": P,
            "grad_eps_mean": ge.sum(0), "grad_J_mean": gJ.sum(0)}


def _exact_density(c, seed):
    n, R = c["N"], c["R"]
    psi = _psi0(c, seed).to(torch.complex128).view(R, n, n)
    rho = torch.zeros(n, n, dtype=torch.complex128, device="cuda")
    for a in (psi.permute(1, 0, 2).reshape(n, -1), psi.permute(2, 0, 1).reshape(n, -1)):
        rho += a @ a.mH
    return {"rho": rho / (2.0 * R)}


def exact(case, seed):
    c = case
    # over about 20 seconds in 64 bits
    if c["kind"] != "density" and work(c)["flops"] * (3.0 if c["kind"] == "adjoint" else 1.0) > 2.5e12:
        return None
    with torch.no_grad():
        if c["kind"] == "density":
            return _exact_density(c, seed)
        if c["kind"] == "adjoint":
            return _exact_adjoint(c, seed)
        if c["kind"] == "graph":
            return _exact_graph(c, seed)
        return _exact_chain(c, seed)
