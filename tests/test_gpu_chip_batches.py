"""Batches of on-chip solves in which gathers fail, against single streaming solves: the gathers that a
solve gives up are solved again in the workspace of the batch, by the passes of its rounding, and the
others keep what they have."""

import math

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

PLAIN, TILE, MARCH = 2, 7, 10


@pytest.fixture(scope="module")
def P():
    import paper_1808_07284_gb300 as pkg
    assert torch.cuda.is_available()
    return pkg


def pairs(sizes, seed):
    out = []
    for i, (nr, nt) in enumerate(sizes):
        obs, pred = synth.gather_pair_hyperbolic(nt=nt, nr=nr, seed=seed + i)
        noise = 0.05 * np.random.default_rng(seed + i).standard_normal(obs.shape).astype(np.float32)
        out.append((torch.from_numpy(obs).cuda(), torch.from_numpy(pred + noise).cuda()))
    return [o for o, _ in out], [p for _, p in out]


def unit(sizes):
    return [1.0 / (nt - 1) for _, nt in sizes], [1.0 / max(nr - 1, 1) for nr, _ in sizes]


def streaming(sizes):
    if max(nr for nr, _ in sizes) <= 8 or all(nr * nt <= 7168 for nr, nt in sizes):
        return PLAIN
    return TILE if sum(nr * nt for nr, nt in sizes) < 1.4e6 else MARCH


def same(got, ref, what):
    """Equal iterates (but for a decision that sums of another order take otherwise, of which there is
    none in these few iterations), and distances of two float sums of equal terms."""
    (d, phi, m, info), (d0, phi0, m0, info0) = got, ref
    assert info["status"] == info0["status"] and info["iters"] == info0["iters"], what
    assert info["ls_trials"] == info0["ls_trials"], what
    for a, b, name in ((phi, phi0, "phi"), (m, m0, "m")):
        rel = float((a.double() - b.double()).norm() / b.double().norm().clamp_min(1e-300))
        assert rel <= 1e-6, (what, name, rel)
    assert math.isclose(d, d0, rel_tol=1e-6), (what, d, d0)


BATCHES = [[(20, 200)] * 4, [(64, 256)] * 4, [(353, 4001)] * 3, [(640, 5000), (64, 256), (300, 5041)],
           [(64, 256), (400, 3000), (20, 8000), (700, 9000), (33, 401)]]


@pytest.mark.parametrize("sizes", BATCHES)
@pytest.mark.parametrize("bad", ["first", "last", "all but one"])
def test_failed_gathers_leave_the_others_alone(P, sizes, bad):
    obs, pred = pairs(sizes, 20)
    dts, dxs = unit(sizes)
    n = len(sizes)
    broken = {"first": [0], "last": [n - 1], "all but one": [b for b in range(n) if b != 1]}[bad]
    for b in broken:
        pred[b] = pred[b].clone()
        pred[b][1, 17] = float("nan")
    d, phis, ms, infos = P.emd_batched(obs, pred, dts, dxs, max_iter=20, check=False)
    assert any(i["tile"] == 0 for b, i in enumerate(infos) if b not in broken)
    for b in range(n):
        if b in broken:
            assert infos[b]["status"] == P.EMD_ERR_NONFINITE
            continue
        ref = P.emd(obs[b], pred[b], dts[b], dxs[b], max_iter=20, tile=infos[b]["tile"] or streaming(sizes))
        same((d[b], phis[b], ms[b], infos[b]), ref, (sizes[b], bad))


@pytest.mark.parametrize("sizes", BATCHES)
def test_failed_linesearches_leave_what_the_passes_of_their_rounding_leave(P, sizes):
    """One trial a decision from small steps: a few iterations pass, then the linesearch gives up.  phi and m
    are the iterates of the streaming passes of the batch's rounding there (those of the tile and the
    marching pass differ by then), and every gather has its trace."""
    obs, pred = pairs(sizes, 40)
    dts, dxs = unit(sizes)
    n, iters = len(sizes), 60
    kw = dict(max_iter=iters, ls_max_trials=1, alpha0=1e-7, check=False)
    tile = streaming(sizes)
    chip = [i["tile"] == 0 for i in P.emd_batched(obs, pred, dts, dxs, max_iter=2)[3]]
    d, phis, ms, infos = P.emd_batched(obs, pred, dts, dxs, **kw)
    failed = 0
    for b in range(n):
        if not chip[b]:
            continue
        ref = P.emd(obs[b], pred[b], dts[b], dxs[b], tile=tile, **kw)
        assert infos[b]["status"] == ref[3]["status"]
        failed += ref[3]["status"] == P.EMD_ERR_LINESEARCH and ref[3]["iters"] > 0
        same((d[b], phis[b], ms[b], infos[b]), ref, sizes[b])
        assert torch.equal(phis[b], ref[1]) and torch.equal(ms[b], ref[2]), sizes[b]
    assert failed
    trace = torch.zeros((n, iters, 4), dtype=torch.float64, device="cuda")
    infos = P.emd_batched(obs, pred, dts, dxs, trace=trace, **kw)[3]
    for b in range(n):
        one = torch.zeros((1, iters, 4), dtype=torch.float64, device="cuda")
        ref = P.emd(obs[b], pred[b], dts[b], dxs[b], tile=tile, trace=one, **kw)[3]
        assert infos[b]["iters"] == ref["iters"]
        k = infos[b]["iters"]
        assert torch.allclose(trace[b, :k], one[0, :k], rtol=1e-5, atol=0.0), sizes[b]


@pytest.mark.parametrize("sizes,tol", [([(64, 256), (40, 300), (100, 400), (64, 256), (12, 700), (33, 401)], 0.1),
                                       ([(64, 256)] * 40, 0.1), ([(200, 2000)] * 6, 0.3),
                                       ([(640, 5000), (300, 5041), (353, 4001)], 0.2),
                                       ([(64, 256), (400, 3000), (700, 9000), (33, 401)], 0.5)])
def test_gathers_of_a_batch_stop_by_themselves(P, sizes, tol):
    """Gathers that stop at a tolerance while their neighbours, and the waves after them, go on: passes
    with a stopping test take the FP64 exchange between others of the fixed-point one, and the streamed
    part of a split batch is dealt again."""
    obs, pred = pairs(sizes, 60)
    for b in range(len(sizes)):  # predicted gathers from near to far from the observed ones
        pred[b] = obs[b] + (0.02 + b / len(sizes)) * (pred[b] - obs[b])
        obs[b] = obs[b] * (1.0 - 0.3 * (b % 3))
    dts, dxs = unit(sizes)
    kw = dict(max_iter=4000, tol=tol, check_every=5)
    d, phis, ms, infos = P.emd_batched(obs, pred, dts, dxs, **kw)
    assert sum(i["tile"] == 0 for i in infos) >= len(sizes) - 1
    assert len({i["iters"] for i in infos}) > 1 and min(i["iters"] for i in infos) < 4000
    for b in range(len(sizes)):
        ref = P.emd(obs[b], pred[b], dts[b], dxs[b], tile=infos[b]["tile"] or streaming(sizes), **kw)
        same((d[b], phis[b], ms[b], infos[b]), ref, (b, sizes[b]))


def test_solves_of_two_threads_at_a_time(P):
    """Two threads with a stream and a workspace each: cooperative launches wait for one another on the
    device, and neither solve sees the other's state."""
    import threading
    sizes = [[(64, 256), (400, 3000)], [(353, 4001), (33, 401)]]
    work = []
    for i, s in enumerate(sizes):
        obs, pred = pairs(s, 80 + 10 * i)
        dts, dxs = unit(s)
        work.append((obs, pred, dts, dxs, P.emd_batched(obs, pred, dts, dxs, max_iter=30)))
    torch.cuda.synchronize()
    errors, gate = [], threading.Barrier(2)

    def run(obs, pred, dts, dxs, ref):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                gate.wait(60)
                for _ in range(20):
                    got = P.emd_batched(obs, pred, dts, dxs, max_iter=30)
                    for b in range(len(obs)):
                        same([g[b] for g in got], [r[b] for r in ref], b)
        except BaseException as e:
            errors.append(e)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
