"""GPU checks of the pairing of heavy with light replicas in batches of more
replicas than SMs: the order a launch deals them in follows the attempts per hop
of the state it runs, never those of a state that has been replaced, and the
pairing changes no chain (hop pairs, cubic lattices, several sides in one handle
and replayed graphs against the oracle, bit for bit).
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_5026_gb300 import build, binding
    build.build()
    binding.load()
    return binding


@pytest.fixture(scope="module")
def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _bits(a):
    return np.ascontiguousarray(a, dtype=np.float64).view(np.uint64)


BASE = dict(nu=0.5, W=1.0, xi=1.0, r_max=3, E=0.01)


def _by_falling(cost):
    # ties in replica order, as the kernel breaks them
    return np.lexsort((np.arange(len(cost)), -cost))


def _rate(a, b):
    # attempts per hop in binary32, as the device keeps it
    d = b["attempts"] - a["attempts"], b["hops"] - a["hops"]
    return d[0].astype(np.float32) / d[1].astype(np.float32)


def test_order_follows_the_state(B, sms):
    R = sms + 40
    s = B.System([dict(BASE, L=8, T=0.03 + 0.002 * (k % 37), seed=k, replica=k)
                  for k in range(R)], precision=B.CG_FP64)
    try:
        start = s.read_group(0)
        # nothing known yet
        np.testing.assert_array_equal(B.cg_debug_schedule(s.h, 0), np.arange(R))
        assert s.run(64, 256) == B.CG_OK
        mid = s.read_group(0)
        assert s.run(64, 256) == B.CG_OK
        end = s.read_group(0)
        # the last launch's attempts per hop
        np.testing.assert_array_equal(B.cg_debug_schedule(s.h, 0),
                                      _by_falling(_rate(mid[2], end[2])))
        # another state: its own counters
        cnt = end[2].copy()
        cnt["hops"] = 100
        cnt["attempts"] = 1000 + 7919 * np.arange(R) % 100003
        s.write_group(0, mid[0], mid[1], cnt)
        want = _by_falling(cnt["attempts"].astype(np.float32) / np.float32(100))
        np.testing.assert_array_equal(B.cg_debug_schedule(s.h, 0), want)
        # the occupations alone replaced: still nothing of the launch before
        s.write_group(0, *mid)
        assert s.run(64, 256) == B.CG_OK
        s.write_group(0, occ=start[0], eps=start[1])
        zero = dict(attempts=np.zeros(R), hops=np.zeros(R))
        c = s.read_group(0, False, False, True)[2]
        np.testing.assert_array_equal(B.cg_debug_schedule(s.h, 0), _by_falling(_rate(zero, c)))
        # and a state without hops: replica order
        s.write_group(0, *start)
        np.testing.assert_array_equal(B.cg_debug_schedule(s.h, 0), np.arange(R))
    finally:
        s.close()


def test_groups_that_run_in_order_have_no_schedule(B):
    s = B.System([dict(BASE, L=8, T=0.1, seed=1)], precision=B.CG_FP64)
    try:
        with pytest.raises(B.CgError):
            B.cg_debug_schedule(s.h, 0)
        with pytest.raises(B.CgError):
            B.cg_debug_schedule(s.h, 1)
    finally:
        s.close()


@pytest.mark.parametrize("form", ["pairs", "cubic", "cubic_pairs", "sides", "graph"])
def test_paired_replicas_run_their_chains(B, sms, form):
    R = sms + 9
    dim = 3 if form.startswith("cubic") else 2
    pair = dict(pair_frac=0.3, pair_rmax=3) if form.endswith("pairs") else {}
    sides = [8] * R + ([12] * R if form == "sides" else [])
    reps = [dict(BASE, L=L, T=0.05 + 0.001 * (k % 50), seed=k, replica=k, dim=dim)
            for k, L in enumerate(sides)]
    s = B.System(reps, precision=B.CG_FP64, use_graph=int(form == "graph"), **pair)
    try:
        for _ in range(3):
            assert s.run(40, 256) == B.CG_OK
        for k in range(len(reps)):
            assert s.observables(k)["hops"] == 120
        for k in (0, 1, sms - 1, sms, R - 1, len(reps) - 2, len(reps) - 1):
            p = reps[k]
            ch = oracle.Chain(p["L"], nu=0.5, W=1.0, xi=1.0, r_max=3, T=p["T"], E=0.01,
                              seed=p["seed"], replica=k, dim=dim, **pair)
            for _ in range(3):
                ch.run(40, 256)
            n, eps, _, cnt = s.state(k)
            on, oeps, _ = ch.state()
            np.testing.assert_array_equal(n, on)
            np.testing.assert_array_equal(_bits(eps), _bits(oeps))
            for f in ("rounds", "hops", "attempts", "P"):
                assert cnt[f] == ch.counters()[f], f
    finally:
        s.close()
