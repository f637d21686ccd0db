"""The work a user has this library do, as cases that can be timed: (T) energies through the public entry points.

Sizes span what the library's own workloads, tests and serving stream use: occupied orbitals from 6 to a few
dozen, v / o between 6 and 13, tiles and K extents that do not divide evenly.  Inputs have the distributions
of the synthetic workloads: integrals from a density-fitting factor B ~ N(0, 0.05) on a 2^-20 grid with
Q = 3 (o + v), sorted uniform orbital energies, t1 ~ N(0, 0.005), t2 ~ N(0, 0.01) with t_ij^ab = t_ji^ba.
"""
import functools
import math

import numpy as np
import torch

import paper_2512_01055_gb300 as tc

DEV = "cuda"


def listed():
    return [
        # A small molecule in FP64, the default precision: latency, launches and tables weigh most.
        {"name": "fp64_tiny", "kind": "dev", "prec": 0, "s": 0, "o": 6, "v": 36},
        # An ordinary small FP64 energy at odd sizes (ragged tiles, ragged K).
        {"name": "fp64_ragged", "kind": "dev", "prec": 0, "s": 0, "o": 9, "v": 77},
        # A whole FP64 energy of a second: the reference-quality number a user compares against.
        {"name": "fp64_large", "kind": "dev", "prec": 0, "s": 0, "o": 12, "v": 132},
        # FP64 contributions of listed triplets of a larger job: spot checks, resuming by triplet range.
        {"name": "fp64_triplets", "kind": "triplets", "prec": 0, "s": 0, "o": 20, "v": 200, "n": 16},
        # The same small molecule on the split path at its default slice count.
        {"name": "split3_tiny", "kind": "dev", "prec": 1, "s": 3, "o": 6, "v": 36},
        # The coarsest split at odd sizes.
        {"name": "split2_ragged", "kind": "dev", "prec": 1, "s": 2, "o": 13, "v": 131},
        # The ordinary single solve, default slices.
        {"name": "split3_single", "kind": "dev", "prec": 1, "s": 3, "o": 20, "v": 200},
        # The finest split.
        {"name": "split4_mid", "kind": "dev", "prec": 1, "s": 4, "o": 15, "v": 172},
        # The largest solve: seconds of tensor-core work, two N chunks.
        {"name": "split3_large", "kind": "dev", "prec": 1, "s": 3, "o": 24, "v": 280},
        # Integrals given as density-fitting factors and assembled on the device.
        {"name": "df_split3", "kind": "df", "prec": 1, "s": 3, "o": 16, "v": 160},
        # The host entry point from page-locked arrays: copies in, energies out.
        {"name": "host_split3", "kind": "host", "prec": 1, "s": 3, "o": 16, "v": 176},
        # A burst of uneven requests to the service, half FP64 and half split, inputs resident.
        {"name": "serve_mix", "kind": "serve", "prec": 0, "s": 3, "o": 6, "v": 10, "n": 12},
    ]


def _flops(o, v):
    return 2.0 * (float(o) ** 3 * float(v) ** 4 + float(o) ** 4 * float(v) ** 3)


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case: a kind of call, o over its range by logarithm, v between 6 and 13 times o."""
    kind = rng.choice(["fp64", "fp64", "triplets", "split", "split", "split", "df", "host", "serve"])
    if kind == "serve":
        lo = rng.randint(5, 7)
        return {"kind": "serve", "prec": 0, "s": rng.choice([2, 3, 4]), "o": lo, "v": lo + rng.randint(1, 3),
                "n": rng.randint(4, 12)}
    while True:
        top = {"fp64": 12, "triplets": 24, "df": 20, "host": 20, "split": 24}[kind]
        o = int(round(_log(rng, 5, top)))
        v = int(round(o * rng.uniform(6.0, 13.0)))
        most = {"fp64": 1.1e12, "df": 2.5e13, "host": 2.5e13, "split": 1.7e14}.get(kind, math.inf)
        if v <= 290 and _flops(o, v) <= most:
            break
    if kind == "triplets":
        each = 12.0 * v ** 4 + 12.0 * o * v ** 3
        return {"kind": "triplets", "prec": 0, "s": 0, "o": o, "v": v,
                "n": rng.randint(1, max(1, min(24, int(7e11 / each))))}
    if kind == "fp64":
        return {"kind": "dev", "prec": 0, "s": 0, "o": o, "v": v}
    return {"kind": "dev" if kind == "split" else kind, "prec": 1, "s": rng.choice([2, 3, 3, 4]), "o": o, "v": v}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _inputs(o, v, seed, salt=0, blocks=True):
    """Device float64 tensors of one job; with blocks the integrals are formed from the factor."""
    g = _gen(seed, salt)
    N, Q = o + v, 3 * (o + v)
    eo = torch.sort(-1.5 + 1.2 * torch.rand(o, generator=g, device=DEV, dtype=torch.float64)).values
    ev = torch.sort(0.1 + 2.9 * torch.rand(v, generator=g, device=DEV, dtype=torch.float64)).values
    x = torch.randn(Q, N, N, generator=g, device=DEV, dtype=torch.float64) * 0.05
    x = torch.triu(torch.clamp(torch.round(x * 2.0 ** 20) * 2.0 ** -20, -0.5, 0.5))
    B = (x + torch.triu(x, 1).transpose(1, 2)).contiguous()
    t1 = torch.randn(o, v, generator=g, device=DEV, dtype=torch.float64) * 0.005
    y = torch.triu(torch.randn(o * v, o * v, generator=g, device=DEV, dtype=torch.float64) * 0.01)
    t2 = (y + torch.triu(y, 1).T).reshape(o, v, o, v).permute(0, 2, 1, 3).contiguous()
    d = {"eps": torch.cat([eo, ev]), "t1": t1, "t2": t2, "B": B}
    if blocks:
        Bov, Bvv, Boo = (B[:, :o, o:].reshape(Q, o * v), B[:, o:, o:].reshape(Q, v * v), B[:, :o, :o].reshape(Q, o * o))
        d["ovvv"] = (Bov.T @ Bvv).reshape(o, v, v, v)
        d["ovoo"] = (Bov.T @ Boo).reshape(o, v, o, o)
        d["ovov"] = (Bov.T @ Bov).reshape(o, v, o, v)
        del d["B"]
    return d


def _triplets(case, seed):
    """n occupied triplets i >= j >= k, not all equal, the last orbital's among them."""
    o = case["o"]
    r = np.random.default_rng(int(seed) % (1 << 32))
    out = [(o - 1, o - 2, 0)]
    while len(out) < case["n"]:
        t = tuple(sorted((int(z) for z in r.integers(0, o, 3)), reverse=True))
        if t[0] != t[2]:
            out.append(t)
    return out


def _requests(case):
    """(o, v, prec, slices) of a burst: sizes cycle through [o, v], precisions alternate."""
    lo, hi = case["o"], case["v"]
    out = []
    for r in range(case["n"]):
        o = lo + (r + r // 3) % (hi - lo + 1)
        v = int(round(o * (6.0 + (7 * r % 11) * 0.3)))
        out.append((o, v, r % 2, case["s"] if r % 2 else 0))
    return out


@functools.lru_cache(maxsize=1)
def _context():
    """One context per process, as a program keeps it."""
    return tc.tc_init(0)


def prepare(case, seed):
    st = {"case": case, "ctx": _context()}
    o, v, kind = case["o"], case["v"], case["kind"]
    if kind == "serve":
        st["jobs"] = [(r, _inputs(r[0], r[1], seed, 1 + n)) for n, r in enumerate(_requests(case))]
        return st
    d = _inputs(o, v, seed, blocks=kind != "df")
    if kind == "host":
        st["pinned"] = [d[k].cpu().pin_memory() for k in ("eps", "t1", "t2", "ovvv", "ovoo", "ovov")]
        st["host"] = [t.numpy() for t in st["pinned"]]
        st["e_ijk"] = np.zeros((o, o, o))
        return st
    st.update(d)
    if kind == "triplets":
        st["trip"] = _triplets(case, seed)
    else:
        st["e_ijk"] = torch.zeros(o, o, o, device=DEV, dtype=torch.float64)
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    o, v, prec, s, kind = case["o"], case["v"], case["prec"], case["s"], case["kind"]
    if kind == "serve":
        tickets = [tc.tc_submit(ctx, r[0], r[1], d["eps"], d["t1"], d["t2"], d["ovvv"], d["ovoo"], d["ovov"],
                                prec=r[2], slices=r[3], device_inputs=True) for r, d in st["jobs"]]
        done = [tc.tc_wait(ctx, t, 60000) for t in tickets]
        if any(code != tc.TC_OK for code, _ in done):
            raise RuntimeError("a request failed: %s" % [code for code, _ in done])
        return {"e_t": np.array([r.e_t for _, r in done]), "e_t5": np.array([r.e_t5 for _, r in done])}
    if kind == "triplets":
        e, r = tc.tc_triplets_dev(ctx, o, v, st["eps"], st["t1"], st["t2"], st["ovvv"], st["ovoo"], st["ovov"],
                                  st["trip"], prec=prec, slices=s)
        return {"e_t": r.e_t, "e_t5": r.e_t5, "e": e}
    if kind == "host":
        eps, t1, t2, ovvv, ovoo, ovov = st["host"]
        r = tc.tc_energy(ctx, o, v, eps, t1, t2, ovvv, ovoo, ovov, prec=prec, slices=s, e_ijk=st["e_ijk"])
    elif kind == "df":
        r = tc.tc_energy_df_dev(ctx, o, v, st["B"], st["eps"], st["t1"], st["t2"], prec=prec, slices=s,
                                e_ijk=st["e_ijk"])
    else:
        r = tc.tc_energy_dev(ctx, o, v, st["eps"], st["t1"], st["t2"], st["ovvv"], st["ovoo"], st["ovov"], prec=prec,
                             slices=s, e_ijk=st["e_ijk"])
    return {"e_t": r.e_t, "e_t5": r.e_t5, "e_ijk": st["e_ijk"]}


def _in_bytes(o, v):
    return 8.0 * (o + v + o * v + 2.0 * o * o * v * v + float(o) * v ** 3 + float(o) ** 3 * v)


def work(case):
    """Inputs read once, results written once; the W contractions of the energy, 2 (o^3 v^4 + o^4 v^3)."""
    o, v = case["o"], case["v"]
    if case["kind"] == "serve":
        reqs = _requests(case)
        return {"bytes": sum(_in_bytes(r[0], r[1]) + 16 for r in reqs), "flops": sum(_flops(r[0], r[1]) for r in reqs)}
    if case["kind"] == "triplets":
        return {"bytes": min(1.0, 3.0 * case["n"] / o) * _in_bytes(o, v) + 8.0 * case["n"],
                "flops": case["n"] * (12.0 * v ** 4 + 12.0 * o * v ** 3)}
    if case["kind"] == "df":
        q, n = 3 * (o + v), o + v
        return {"bytes": 8.0 * (q * n * n + n + o * v + float(o * v) ** 2 + o ** 3),
                "flops": _flops(o, v) + 2.0 * q * o * v * (v * v + o * o + o * v)}
    return {"bytes": _in_bytes(o, v) + 8.0 * o ** 3, "flops": _flops(o, v)}


# ---------------------------------------------------------------------------
# The same numbers from plain 64-bit torch
# ---------------------------------------------------------------------------

def _triplet_exact(d, i, j, k):
    """(weighted energy, its V part) of one occupied triplet i >= j >= k."""
    o, v = d["t1"].shape
    ovvv, t2, ovoo, ovov, t1, eps = d["ovvv"], d["t2"], d["ovoo"], d["ovov"], d["t1"], d["eps"]

    def x(p, q, r):     # sum_f (pa|bf) t_rq^cf - sum_l (pa|ql) t_lr^bc, over [a, b, c]
        part = (ovvv[p].reshape(v * v, v) @ t2[r, q].T).reshape(v, v, v)
        return part - (ovoo[p, :, q, :] @ t2[:, r].reshape(o, v * v)).reshape(v, v, v)

    W = x(i, j, k)
    W = W + x(i, k, j).permute(0, 2, 1)
    W = W + x(j, i, k).permute(1, 0, 2)
    W = W + x(j, k, i).permute(2, 0, 1)
    W = W + x(k, j, i).permute(2, 1, 0)
    W = W + x(k, i, j).permute(1, 2, 0)
    V = (t1[i][:, None, None] * ovov[j, :, k, :][None] + t1[j][None, :, None] * ovov[i, :, k, :][:, None, :]
         + t1[k][None, None, :] * ovov[i, :, j, :][:, :, None])
    ev = eps[o:]
    D = (eps[i] + eps[j] + eps[k]) - (ev[:, None, None] + ev[None, :, None] + ev[None, None, :])
    Y = 4.0 * W + W.permute(1, 2, 0) + W.permute(2, 0, 1) - 2.0 * (W.permute(1, 0, 2) + W.permute(0, 2, 1)
                                                                  + W.permute(2, 1, 0))
    Y = Y / D
    w = 2 - (i == j) - (j == k)
    e5 = (V * Y).sum()
    return w * ((W * Y).sum() + e5), w * e5


def _all_triplets(o):
    return [(i, j, k) for i in range(o) for j in range(i + 1) for k in range(j + 1) if i != k]


def _energy_exact(d, trip):
    pairs = [_triplet_exact(d, *t) for t in trip]
    e = torch.stack([p[0] for p in pairs]).cpu().numpy()
    return e, math.fsum(e.tolist()), math.fsum(torch.stack([p[1] for p in pairs]).cpu().tolist())


def exact(case, seed):
    o, v, kind = case["o"], case["v"], case["kind"]
    if work(case)["flops"] > 8e12:
        return None
    if kind == "serve":
        both = []
        for n, r in enumerate(_requests(case)):
            d = _inputs(r[0], r[1], seed, 1 + n)
            both.append(_energy_exact(d, _all_triplets(r[0]))[1:])
        return {"e_t": np.array([b[0] for b in both]), "e_t5": np.array([b[1] for b in both])}
    d = _inputs(o, v, seed)
    trip = _triplets(case, seed) if kind == "triplets" else _all_triplets(o)
    e, e_t, e_t5 = _energy_exact(d, trip)
    if kind == "triplets":
        return {"e_t": e_t, "e_t5": e_t5, "e": e}
    e_ijk = np.zeros((o, o, o))
    for t, val in zip(trip, e):
        e_ijk[t] = val
    return {"e_t": e_t, "e_t5": e_t5, "e_ijk": e_ijk if kind == "host" else torch.from_numpy(e_ijk)}
