"""The on-chip solve (default for gathers whose state fits in the GPU's shared and tensor memory)
against the streaming pass of the same rounding (the tile pass below 1.4 million cells, the marching
pass above) on the same inputs, at the sizes where its layout can go wrong: runs of one row per
warp, one row more, the tallest CTA and the first that needs a second segment, tall CTAs, strips of
120 samples and their remainders, receivers and samples at the ends of the range.

The two paths do the same arithmetic on every cell, in the same order, so phi and m may differ
only where a linesearch decision differs; the sums behind the decisions are added in another
order, which moves the reported residual by FP32 rounding of partial sums (a few 1e-8).  Physical
spacings keep the receiver flux shut for the first iterations; the unit square opens both."""

import math

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

DT, DX = 2e-3, 10.0
TILE = 7      # the TMA tile pass
PLAIN = 2     # the plain pass (any number of receivers)
MARCH = 10    # the marching pass


def streaming(cells, nr):
    return PLAIN if nr <= 8 else TILE if cells < 1.4e6 else MARCH


def spacings(nr, nt):
    return [(DT, DX), (1.0 / (nt - 1), 1.0 / max(nr - 1, 1))]


@pytest.fixture(scope="module")
def P():
    import paper_1808_07284_gb300 as pkg
    assert torch.cuda.is_available()
    return pkg


def pair(nr, nt, seed=0):
    obs, pred = synth.gather_pair_hyperbolic(nt=nt, nr=nr, seed=seed)
    rng = np.random.default_rng(seed + 1)
    noise = 0.05 * rng.standard_normal(obs.shape).astype(np.float32)
    return torch.from_numpy(obs).cuda(), torch.from_numpy(pred + noise).cuda()


def check(got, ref, what=""):
    d, phi, m, info = got
    d0, phi0, m0, info0 = ref
    assert info["status"] == 0 and info0["status"] == 0, what
    assert info["iters"] == info0["iters"] and info["ls_trials"] == info0["ls_trials"], what
    for a, b, name in ((phi, phi0, "phi"), (m, m0, "m")):
        rel = float((a.double() - b.double()).norm() / b.double().norm().clamp_min(1e-300))
        assert rel <= 1e-6, (what, name, rel)
    for key in ("dist_l1", "residual", "duality_gap"):
        assert math.isclose(info[key], info0[key], rel_tol=1e-5, abs_tol=1e-12), (what, key)
    for key in ("mass_mu", "mass_nu"):
        assert math.isclose(info[key], info0[key], rel_tol=1e-12), (what, key)


SHAPES = [(64, 256), (12, 700), (13, 700), (27, 400), (28, 400), (125, 120), (126, 121), (250, 1000),
          (251, 999), (9, 1201), (2, 4801), (3, 2399), (1, 9001), (640, 61), (648, 1201), (400, 3000),
(480, 4000), (353, 4001), (648, 2761), (9, 156001), (300, 5041), (648, 8000)]


@pytest.mark.parametrize("norm", [1, 2])
@pytest.mark.parametrize("nr,nt", SHAPES)
def test_matches_the_streaming_pass(P, nr, nt, norm):
    o, p = pair(nr, nt)
    tile = streaming(nr * nt, nr)
    for dt, dx in spacings(nr, nt):
        kw = dict(norm=norm)
        got, ref = P.emd(o, p, dt, dx, max_iter=25, **kw), P.emd(o, p, dt, dx, max_iter=25, tile=tile, **kw)
        if (nr, nt) != (9, 156001):  # more strips than SMs: streams
            assert got[3]["tile"] == 0 and got[3]["launches"] == 1  # on chip
        check(got, ref)
        # from a warm start, in place, and on a single iteration
        kw.update(phi_init=ref[1], m_init=ref[2])
        check(P.emd(o, p, dt, dx, max_iter=9, **kw), P.emd(o, p, dt, dx, max_iter=9, tile=tile, **kw), "warm")
        check(P.emd(o, p, dt, dx, max_iter=1, **kw), P.emd(o, p, dt, dx, max_iter=1, tile=tile, **kw), "one")


@pytest.mark.parametrize("scale", [1e-12, 1e-6, 1e4, 1e8])
@pytest.mark.parametrize("nr,nt", [(64, 256), (353, 4001)])
def test_amplitudes_match_the_streaming_pass(P, nr, nt, scale):
    """Sums below 2^-60 and above 2^60 take the FP64 exchange in every pass, the others the
    fixed-point one."""
    o, p = pair(nr, nt, seed=4)
    o, p = o * scale, p * scale
    tile = streaming(nr * nt, nr)
    for dt, dx in spacings(nr, nt):
        check(P.emd(o, p, dt, dx, max_iter=25), P.emd(o, p, dt, dx, max_iter=25, tile=tile), (nr, nt, scale, dt))


@pytest.mark.parametrize("kw", [dict(norm=2), dict(balance=0), dict(linesearch=0), dict(tol=1e-30, check_every=7),
                                dict(xi=0.9), dict(alpha0=1e-3)])
def test_options_match_the_streaming_pass(P, kw):
    for nr, nt in ((70, 500), (300, 4700), (420, 5000)):
        o, p = pair(nr, nt, seed=3)
        tile = streaming(nr * nt, nr)
        for dt, dx in spacings(nr, nt):
            check(P.emd(o, p, dt, dx, max_iter=30, **kw), P.emd(o, p, dt, dx, max_iter=30, tile=tile, **kw), str(kw))


def test_tolerance_stop_and_trace(P):
    o, p = pair(40, 300, seed=4)
    dt, dx = 1.0 / 299, 1.0 / 39
    tr = [torch.zeros((1, 3000, 4), dtype=torch.float64, device="cuda") for _ in range(2)]
    got = P.emd(o, p, dt, dx, max_iter=3000, tol=0.3, trace=tr[0])
    ref = P.emd(o, p, dt, dx, max_iter=3000, tol=0.3, trace=tr[1], tile=TILE)
    assert 10 <= got[3]["iters"] < 3000
    check(got, ref)
    assert torch.equal(tr[0][..., 2], tr[1][..., 2])
    assert torch.allclose(tr[0], tr[1], rtol=1e-5, atol=0.0)


def test_unaligned_inputs_and_outputs(P):
    nr, nt = 33, 402
    o, p = pair(nr, nt, seed=5)
    def shifted(t, planes=1):
        buf = torch.zeros(planes * nr * nt + 1, device="cuda")
        v = buf[1:].view((planes, nr, nt) if planes > 1 else (nr, nt))
        if t is not None:
            v.copy_(t)
        return v
    phi, m = shifted(None), shifted(None, 2)
    ws = P.new_workspace(P.emd_workspace_size(nt, nr), o.device)
    res = P.emd_dyn_solve(shifted(o), shifted(p), DT, DX, P.emd_default_params(max_iter=40), phi, m, ws)
    check((res.dist, phi, m, res.as_dict()), P.emd(o, p, DT, DX, max_iter=40, tile=TILE))


def test_batch_of_uneven_gathers_one_too_large(P):
    sizes = [(64, 256), (400, 3000), (20, 8000), (700, 9000), (33, 401), (200, 1500)]
    pairs = [pair(nr, nt, seed=10 + i) for i, (nr, nt) in enumerate(sizes)]
    obs, pred = [a for a, _ in pairs], [b for _, b in pairs]
    d, phis, ms, infos = P.emd_batched(obs, pred, DT, DX, max_iter=30)
    assert [i["tile"] == 0 for i in infos].count(True) >= 5
    total = sum(nr * nt for nr, nt in sizes)
    for b, (nr, nt) in enumerate(sizes):
        ref = P.emd(obs[b], pred[b], DT, DX, max_iter=30, tile=infos[b]["tile"] or streaming(total, 9))
        check((d[b], phis[b], ms[b], infos[b]), ref, str(sizes[b]))


def test_failures_come_back_as_the_streaming_solve_reports_them(P):
    o, p = pair(64, 256)
    bad = p.clone()
    bad[10, 17] = float("nan")
    for kw in (dict(), dict(tile=TILE)):
        _, _, _, info = P.emd(o, bad, DT, DX, max_iter=20, check=False, **kw)
        assert info["status"] == P.EMD_ERR_NONFINITE
        _, phi, m, info = P.emd(o, p, DT, DX, max_iter=20, check=False, debug_fault=1, **kw)
        assert info["status"] == P.EMD_ERR_LINESEARCH and info["iters"] == 0
        assert bool(torch.isfinite(phi).all()) and bool(torch.isfinite(m).all())
    # a batch reports each gather by itself
    d, _, _, infos = P.emd_batched([o, o], [bad, p], DT, DX, max_iter=20, check=False)
    assert infos[0]["status"] == P.EMD_ERR_NONFINITE and infos[1]["status"] == 0
    check((d[1], None, None, infos[1])[:1] + P.emd(o, p, DT, DX, max_iter=20)[1:], P.emd(o, p, DT, DX, max_iter=20, tile=TILE))


def test_a_wait_that_runs_out_is_reported(P):
    o, p = pair(64, 256)
    _, _, _, info = P.emd(o, p, DT, DX, max_iter=20, check=False, debug_fault=2)
    assert info["status"] == P.EMD_ERR_TIMEOUT
    check(P.emd(o, p, DT, DX, max_iter=20), P.emd(o, p, DT, DX, max_iter=20, tile=TILE))


@pytest.mark.parametrize("norm", [1, 2])
@pytest.mark.parametrize("nr,nt", [(1, 2), (1, 1024), (1, 7168), (2, 2), (3, 5), (2, 3584), (20, 200), (64, 112),
                                   (7, 1021), (896, 8), (1433, 5), (200, 33)])
def test_small_gathers_match_the_plain_pass(P, nr, nt, norm):
    """The one-CTA solve in shared memory (and, where padding its rows to four samples takes too
    much of it, the on-chip solve): odd rows, single receivers, one quad a row, the largest."""
    o, p = pair(nr, nt, seed=6)
    for dt, dx in spacings(nr, nt):
        kw = dict(norm=norm)
        got, ref = P.emd(o, p, dt, dx, max_iter=40, **kw), P.emd(o, p, dt, dx, max_iter=40, tile=PLAIN, **kw)
        assert got[3]["tile"] == 0
        check(got, ref)
        kw.update(phi_init=ref[1], m_init=ref[2])
        check(P.emd(o, p, dt, dx, max_iter=9, **kw), P.emd(o, p, dt, dx, max_iter=9, tile=PLAIN, **kw), "warm")


def test_small_gathers_stop_trace_and_fail_alike(P):
    o, p = pair(16, 250, seed=7)
    dt, dx = 1.0 / 249, 1.0 / 15
    tr = [torch.zeros((1, 2000, 4), dtype=torch.float64, device="cuda") for _ in range(2)]
    got = P.emd(o, p, dt, dx, max_iter=2000, tol=0.3, trace=tr[0])
    ref = P.emd(o, p, dt, dx, max_iter=2000, tol=0.3, trace=tr[1], tile=PLAIN)
    assert got[3]["iters"] < 2000
    check(got, ref)
    assert torch.equal(tr[0][..., 2], tr[1][..., 2])
    assert torch.allclose(tr[0], tr[1], rtol=1e-5, atol=0.0)
    bad = p.clone()
    bad[3, 17] = float("inf")
    assert P.emd(o, bad, dt, dx, max_iter=20, check=False)[3]["status"] == P.EMD_ERR_NONFINITE
    # a failed solve from a warm start in place reports the same, and leaves what the passes leave
    out = []
    for tile in (0, PLAIN):
        phi, m = ref[1].clone(), ref[2].clone()
        ws = P.new_workspace(P.emd_workspace_size(250, 16), o.device)
        res = P.emd_dyn_solve(o, p, dt, dx, P.emd_default_params(max_iter=20, debug_fault=1, tile=tile, phi_init=phi,
                                                                 m_init=m), phi, m, ws, check=False)
        assert res.status == P.EMD_ERR_LINESEARCH
        out.append((phi, m))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
