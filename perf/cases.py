"""The workloads that the speed of this library is measured on.

Two kinds of pass, each through the public binding as a user's program makes it:

``chain``   the program holds a handle and a checkpoint of its replicas (pinned
            host buffers); a pass restores the checkpoint, advances every
            replica by ``hops`` executed hops, rebuilds binary32 energies from
            their definition, and reads occupations, energies and counters
            back.  The checkpoints are relaxed chains, not random starts.
``resume``  the program holds occupations only; a pass uploads them, rebuilds
            the energies on the device and reads them back.

A handle is built once and kept, as a program that runs for hours keeps it.
The restored energies make each pass the same work whatever ran before it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1407_5026_gb300 import binding as B

CHAIN = dict(kind="chain", precision="fp32", dim=2, sites="lattice", nu=0.5, W=1.0, xi=1.0,
             r_max=6, T=0.05, E=0.01, M=4096, cluster=0, clock="deterministic", pair_frac=0.0,
             pair_rmax=0, graph=False, refresh=True)


def _chain(name, L, R, hops, relax, **kw):
    return dict(CHAIN, name=name, L=L, R=R, hops=hops, relax=relax, **kw)


def listed():
    return [
        # one small binary64 replica: the calls around a short run count most
        _chain("l16_fp64_single", 16, 1, 128, 1024, precision="fp64", r_max=4, E=0.0, M=256,
               refresh=False),
        # the relaxation study: three temperatures times eight disorder seeds
        # in one handle, binary64, the stochastic clock
        _chain("l64_fp64_sweep", 64, 24, 512, 16384, precision="fp64", T=0.02, T_high=0.1,
               clock="gaussian", refresh=False),
        # the flagship: 304 binary32 disorder replicas at low temperature
        _chain("l128_fp32_batch", 128, 304, 1024, 32768, W=2.0, r_max=8, T=0.01, E=0.005),
        # the same system in the bit-exact form, one replica per SM
        _chain("l128_fp64_batch", 128, 152, 128, 24576, precision="fp64", W=2.0, r_max=8, T=0.01,
               E=0.005, refresh=False),
        # a mixed batch of four lattice sizes replayed from a CUDA graph
        _chain("mixed_fp32_graph", 0, 256, 512, 8192, T=0.03, graph=True),
        # a large lattice, each replica on a cluster of four CTAs
        _chain("l256_fp32_cluster", 256, 16, 1024, 49152, xi=1.5, r_max=10, T=0.02, E=0.005,
               M=16384, cluster=4),
        # the cubic lattice, one replica per SM
        _chain("cubic32_fp32", 32, 152, 512, 8192, dim=3, r_max=3),
        # the cubic lattice past one CTA; 48 = 3 * 16 takes the mixed-radix refresh
        _chain("cubic48_fp32_cluster", 48, 16, 256, 4096, dim=3, r_max=3, cluster=4),
        # a fifth of the labels propose two-electron hops
        _chain("l64_fp32_pairs", 64, 304, 512, 8192, pair_frac=0.2, pair_rmax=4),
        # sites at random positions: binary64, the N x N couplings in device memory
        _chain("random64_fp64", 64, 24, 512, 8192, precision="fp64", sites="random",
               refresh=False),
        # resuming the flagship from occupations alone (power-of-two side)
        dict(kind="resume", name="l128_resume", L=128, R=304, dim=2, W=2.0, r_max=8),
        # the same for a side that is neither 2^m nor 3 2^m
        dict(kind="resume", name="l112_resume", L=112, R=128, dim=2, W=1.0, r_max=6),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(x, lo=4):
    return max(lo, 2 * int(round(x / 2)))


def _hops(R, sites, T, lanes, most=1024):
    """Hops that keep a drawn pass below the flagship's: a hop costs its
    N-site update and about 1/(0.03 T) proposals; `lanes` replicas advance
    side by side."""
    per_hop = (sites / 8.0 + 1.0 / (0.03 * T)) * max(1.0, R / lanes)
    return max(16, min(most, int(3.0e6 / per_hop)))


def _most_replicas(R, L, N):
    """Sides without a fast refresh (neither 2^m nor 3 2^m, nor a multiple of
    16) rebuild by N^2 / 2 binary64 adds per replica: fewer replicas."""
    m = L // 3 if L % 3 == 0 else L
    fast = m & (m - 1) == 0 or (L % 16 == 0 and R >= 8)
    return R if fast else max(1, min(R, 64, int(1.0e9 / (N * N / 2.0))))


def draw(rng):
    kind = rng.choice(["square", "square", "square", "cluster", "cubic", "random", "resume"])
    T = round(_log(rng, 0.01, 0.1), 4)
    E = rng.choice([0.0, 0.005, 0.01])
    W = rng.choice([1.0, 2.0])
    if kind == "square":
        fp64 = rng.random() < 0.35
        L = _even(_log(rng, 16, 128))
        R = int(_log(rng, 1, 152 if fp64 else 304))
        R = R if fp64 else _most_replicas(R, L, L * L)
        pair = rng.choice([0.0, 0.0, 0.1, 0.3])
        hops = _hops(R, L * L * (4 if fp64 else 1), T, 152) // (2 if pair else 1)
        return _chain("", L, R, hops, 2048, precision="fp64" if fp64 else "fp32", T=T, E=E, W=W,
                      r_max=rng.choice([4, 6]), M=rng.choice([1024, 4096, 16384]),
                      clock=rng.choice(["deterministic", "deterministic", "gaussian"]),
                      pair_frac=pair, pair_rmax=4 if pair else 0, refresh=not fp64)
    if kind == "cluster":
        C = rng.choice([2, 4, 8])
        L = 16 * rng.randint(8, 16)
        R = rng.choice([1, rng.randint(8, 16)])
        return _chain("", L, R, _hops(R, L * L / C, T, 152 // C), 1024, T=T, E=E, W=W,
                      r_max=rng.choice([6, 8]), M=rng.choice([4096, 16384]),
                      cluster=C if L * L * 4 / C < 150000 else 8)
    if kind == "cubic":
        L = _even(_log(rng, 8, 32))
        R = _most_replicas(int(_log(rng, 1, 152)), L, L ** 3)
        return _chain("", L, R, _hops(R, L ** 3, T, 152), 1024, dim=3, T=T, E=E, W=W, r_max=3)
    if kind == "random":
        L = _even(_log(rng, 16, 64))
        R = rng.randint(1, 24)
        return _chain("", L, R, _hops(R, L * L * 4, T, 152), 1024, precision="fp64",
                      sites="random", T=T, E=E, W=W, r_max=rng.choice([4, 6]), refresh=False)
    dim = rng.choice([2, 2, 3])
    L = _even(_log(rng, 8, 32)) if dim == 3 else 16 * rng.randint(2, 10)
    R = _most_replicas(int(_log(rng, 8, 256)), L, L ** dim)
    return dict(kind="resume", L=L, R=R, dim=dim, W=W, r_max=3)


def _sides(c):
    """The side of each replica (the mixed batch draws them, the same ones each time)."""
    if c["L"]:
        return [c["L"]] * c["R"]
    return [int(x) for x in np.random.default_rng(0).choice([32, 48, 64, 96], size=c["R"])]


def _replicas(c, seed):
    out = []
    for k, L in enumerate(_sides(c)):
        T = c["T"]
        if "T_high" in c:       # a sweep: low, middle (geometric) and high, in turn
            T = (c["T"], 0.05, c["T_high"])[k % 3]
        out.append(dict(L=L, nu=c["nu"], W=c["W"], xi=c["xi"], r_max=c["r_max"], T=T, E=c["E"],
                        seed=seed * 4096 + k, replica=k, dim=c["dim"],
                        sites=B.CG_SITES_RANDOM if c["sites"] == "random" else B.CG_SITES_LATTICE))
    return out


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True).numpy()


class _Group:
    """Pinned checkpoint and result buffers of the replicas of one side."""

    def __init__(self, sysm, g, precision):
        self.idx, N, words = sysm.group_dims(g)
        cnt = len(self.idx)
        ft = torch.float32 if precision == B.CG_FP32 else torch.float64
        bufs = [(_pinned((cnt, words), torch.int32).view(np.uint32), _pinned((cnt, N), ft),
                 np.zeros(cnt, B.COUNTERS_DTYPE)) for _ in range(2)]
        self.start, self.end = bufs


def prepare(case, seed):
    c = dict(case)
    torch.cuda.set_device(0)
    if c["kind"] == "resume":
        reps = [dict(L=c["L"], nu=0.5, W=c["W"], xi=1.0, r_max=c["r_max"], T=0.05, E=0.0,
                     seed=seed * 4096 + k, replica=k, dim=c["dim"]) for k in range(c["R"])]
        sysm = B.System(reps, precision=B.CG_FP32)
        g = _Group(sysm, 0, B.CG_FP32)
        g.start[0][:] = _packed_occupations(c, seed)
        return dict(case=c, sys=sysm, groups=[g])
    precision = B.CG_FP64 if c["precision"] == "fp64" else B.CG_FP32
    sysm = B.System(_replicas(c, seed), precision=precision, use_graph=int(c["graph"]),
                    cluster_size=c["cluster"], pair_frac=c["pair_frac"], pair_rmax=c["pair_rmax"],
                    time_mode=B.CG_TIME_GAUSSIAN if c["clock"] == "gaussian"
                    else B.CG_TIME_DETERMINISTIC)
    sysm.run(c["relax"], c["M"])
    groups = [_Group(sysm, g, precision) for g in range(B.cg_num_groups(sysm.h))]
    for k, g in enumerate(groups):
        sysm.read_group(k, *g.start)
    return dict(case=c, sys=sysm, groups=groups)


def run(state):
    c, sysm, groups = state["case"], state["sys"], state["groups"]
    if c["kind"] == "resume":
        g = groups[0]
        sysm.write_group(0, occ=g.start[0])
        B.cg_refresh_async(sysm.h)
        sysm.read_group(0, False, g.end[1], False)
        return {"eps": g.end[1]}
    for k, g in enumerate(groups):
        sysm.write_group(k, *g.start)
    B.cg_run_async(sysm.h, c["hops"], c["M"])
    if c["refresh"]:
        B.cg_refresh_async(sysm.h)
    B.cg_sync(sysm.h)
    out = {}
    for k, g in enumerate(groups):
        occ, eps, cnt = sysm.read_group(k, *g.end)
        # `evaluated` (labels looked at past the executed one) follows the
        # launch shape and is no result of the chain
        out[str(k)] = {"occ": occ.view(np.int32), "eps": eps, "energy": cnt["energy"],
                       "time": cnt["time"],
                       **{f: cnt[f].astype(np.int64) for f in ("rounds", "hops", "attempts", "P")}}
    return out


def work(case):
    """Bytes: occupations, energies (and, for a refresh, the site energies)
    read once and written once.  Flops: two adds per site and hop for the
    long-range update (proposals are integer work and decide by a compare),
    and 5 N log2 N per real transform pair of a refresh."""
    c = dict(case)
    sides = [c["L"]] * c["R"] if c["L"] else [32, 48, 64, 96] * (c["R"] // 4)
    real = 4 if c.get("precision", "fp32") == "fp32" else 8
    total = dict(bytes=0.0, flops=0.0)
    for L in sides:
        N = L ** c["dim"]
        fft = 5.0 * N * math.log2(N)
        if c["kind"] == "resume":
            total["bytes"] += N / 8 + 8 * N + real * N
            total["flops"] += fft
            continue
        total["bytes"] += 2 * (N / 8 + real * N) + (8 * N if c["refresh"] else 0)
        total["flops"] += 2.0 * N * c["hops"] + (fft if c["refresh"] else 0)
        if c["sites"] == "random":
            # each hop reads two rows of the replica's coupling matrix
            total["bytes"] += 16.0 * N * c["hops"]
    return total


def _occupations(c, seed):
    """(R, N) occupations, half filled, from the seed."""
    N = c["L"] ** c["dim"]
    rng = np.random.default_rng(seed)
    n = np.zeros((c["R"], N), np.uint8)
    n[:, : N // 2] = 1
    return rng.permuted(n, axis=1)


def _packed_occupations(c, seed):
    n = _occupations(c, seed)
    pad = -n.shape[1] % 32
    if pad:
        n = np.concatenate([n, np.zeros((n.shape[0], pad), np.uint8)], axis=1)
    return np.packbits(n, axis=1, bitorder="little").view(np.uint32)


def _site_energies(c, seed, k):
    """phi of replica k: W (u - 1/2), u from word 0 of the Philox-4x32-10 block
    (Salmon et al., SC'11) of counter (s, 1, 2^32 - 1, replica) under the seed."""
    N = c["L"] ** c["dim"]
    m32 = np.uint64(0xFFFFFFFF)
    x = [np.arange(N, dtype=np.uint64), np.full(N, 1, np.uint64), np.full(N, 0xFFFFFFFF, np.uint64),
         np.full(N, k, np.uint64)]
    s = seed * 4096 + k
    k0, k1 = s & 0xFFFFFFFF, s >> 32
    for _ in range(10):
        p0, p1 = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
        x = [(p1 >> np.uint64(32)) ^ x[1] ^ np.uint64(k0), p1 & m32,
             (p0 >> np.uint64(32)) ^ x[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c["W"] * ((x[0].astype(np.float64) + 0.5) * 2.0 ** -32 - 0.5)


def exact(case, seed):
    """Energies of a resume from their definition, phi + (1/r) * (n - 1/2) on
    the torus, in 64 bits.  A chain's outputs follow from its random decisions,
    which no closed form gives."""
    c = dict(case)
    if c["kind"] != "resume":
        return None
    L, dim = c["L"], c["dim"]
    f = np.minimum(np.arange(L), L - np.arange(L)).astype(np.float64)
    r2 = f[:, None] ** 2 + f[None, :] ** 2
    if dim == 3:
        r2 = f[:, None, None] ** 2 + r2[None]
    g = np.zeros_like(r2)
    g[r2 > 0] = 1.0 / np.sqrt(r2[r2 > 0])
    gh = torch.fft.rfftn(torch.from_numpy(g))
    n = torch.from_numpy(_occupations(c, seed)).to(torch.float64).reshape((c["R"],) + (L,) * dim)
    axes = tuple(range(1, dim + 1))
    conv = torch.fft.irfftn(torch.fft.rfftn(n - 0.5, dim=axes) * gh, s=(L,) * dim, dim=axes)
    phi = np.stack([_site_energies(c, seed, k) for k in range(c["R"])])
    return {"eps": phi + conv.reshape(c["R"], -1).numpy()}
