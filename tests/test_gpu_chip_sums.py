"""The balancing sums of the on-chip solve (f, f^2, |Pcal| + |Pobs|, Pcal - Pobs) against exact ones,
in its three forms, at amplitudes whose squares leave the range of FP32.

The sums are added in pairs of floats within a lane, to about 2^-48 of a lane's part, whose errors
average out over the lanes, and in FP64 above it: at most 5 additions in a warp, 4 in a CTA, 19 + 2 across the
CTAs of a copy and the copies, each rounded to 2^-53 of a partial sum, so they are exact to 4e-15 of
the sum of the magnitudes.  Gathers whose sums leave the range of FP32 go back to the streaming solve.  The reported
residual is sqrt(sum p^2) / |f|, whose numerator is a sum of FP32 squares in every solve: 1e-5, as
between any two of them."""

import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

PLAIN, TILE, MARCH = 2, 7, 10
SIZES = [(64, 256), (353, 4001), (640, 5000)]  # the tile form, the marching one, tall CTAs


@pytest.fixture(scope="module")
def P():
    import paper_1808_07284_gb300 as pkg
    assert torch.cuda.is_available()
    return pkg


def noise(nr, nt, seed):
    return np.random.default_rng(seed).standard_normal((nr, nt))


def solve(P, obs, pred, **kw):
    o, p = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda() for a in (obs, pred))
    return P.emd(o, p, 1.0, 1.0, **kw)


@pytest.mark.parametrize("nr,nt", SIZES)
@pytest.mark.parametrize("offset", [0.0, 1e3])
def test_masses_are_exact_to_fp64(P, nr, nt, offset):
    obs = noise(nr, nt, 1).astype(np.float32)
    pred = (noise(nr, nt, 2) + offset).astype(np.float32)
    info = solve(P, obs, pred, max_iter=1)[3]
    assert info["status"] == 0 and info["tile"] == 0
    o, p = obs.astype(np.float64).ravel(), pred.astype(np.float64).ravel()
    total, net = math.fsum(np.abs(o)) + math.fsum(np.abs(p)), math.fsum(p - o)  # p - o is exact in FP64
    bound = 4e-15 * total
    assert abs(info["mass_mu"] + info["mass_nu"] - total) <= bound
    assert abs(info["imbalance"] - net) <= bound


@pytest.mark.parametrize("nr,nt", SIZES)
def test_residual_of_small_amplitudes(P, nr, nt):
    """Squares of 1e-44: a few of FP32's smallest steps, so a norm of f that is summed in FP32 is off
    by a thousandth or more (the numerator's squares are those steps in every solve)."""
    obs, pred = 1e-22 * noise(nr, nt, 3), 1e-22 * noise(nr, nt, 4)
    got = solve(P, obs, pred, max_iter=5, alpha0=1e-4)[3]
    ref = solve(P, obs, pred, max_iter=5, alpha0=1e-4, tile=TILE if nr * nt < 1.4e6 else MARCH)[3]
    assert got["status"] == ref["status"] == 0
    assert math.isclose(got["r_feas"], ref["r_feas"], rel_tol=1e-5), (got["r_feas"], ref["r_feas"])


def check_like_streaming(P, obs, pred):
    nr, nt = obs.shape
    got = solve(P, obs, pred, max_iter=5, alpha0=1e-4)
    ref = solve(P, obs, pred, max_iter=5, alpha0=1e-4, tile=TILE if nr * nt < 1.4e6 else MARCH)
    assert got[3]["status"] == ref[3]["status"] == 0
    for key in ("r_feas", "mass_mu", "mass_nu", "dist"):
        assert math.isclose(got[3][key], ref[3][key], rel_tol=1e-5), (key, got[3][key], ref[3][key])


@pytest.mark.parametrize("nr,nt", SIZES)
def test_residual_above_a_common_level(P, nr, nt):
    """Pcal on a level whose squares FP32 cannot add up.  Balancing takes the level out, so the pass's
    own sums stay in range, and the gather is solved by the streaming passes."""
    check_like_streaming(P, np.zeros((nr, nt)), 8e18 + 1e16 * noise(nr, nt, 5))


@pytest.mark.parametrize("nr,nt", SIZES)
def test_masses_beyond_the_range_of_a_float(P, nr, nt):
    """Equal values of 1e37 in both gathers: f is zero there, but a lane's mass is not a float.  The
    gather goes back to the streaming solve."""
    big = noise(nr, nt, 6) < 0.0
    check_like_streaming(P, np.where(big, 1e37, 0.0), np.where(big, 1e37, noise(nr, nt, 7)))


@pytest.mark.parametrize("nr,nt,tile", [(1, 256, PLAIN), (1, 1024, PLAIN), (20, 200, PLAIN), (64, 256, TILE),
                                        (640, 5000, MARCH)])
def test_reported_residual_is_as_near_to_64_bits_as_the_streaming_one(P, nr, nt, tile):
    """Both round in float32 within a warp and are as good as exact above it, so over many inputs their
    errors have one size; that of 40 inputs is known to about a tenth."""
    rms = []
    for t in (0, tile):
        total = 0.0
        for seed in range(40):
            g = torch.Generator(device="cuda").manual_seed(seed)
            x = torch.nn.functional.avg_pool1d(torch.randn((2, nr, nt), device="cuda", generator=g), 9, 1, 4).contiguous()
            dt, dx = 1.0 / (nt - 1), 1.0 / max(nr - 1, 1)
            _, _, m, info = P.emd(x[0], x[1], dt, dx, max_iter=30, tile=t)
            f = x[1] - x[0]
            balanced = (f - f.double().mean().float()).double()  # as the solve has it
            u = m.double()
            div = torch.diff(u[1], dim=1, append=torch.zeros((nr, 1), device="cuda")) / dt
            if nr > 1:
                div = div + torch.diff(u[0], dim=0, append=torch.zeros((1, nt), device="cuda")) / dx
            exact = float((div + balanced).norm() / (f.double() - f.double().mean()).norm())
            total += (info["r_feas"] / exact - 1.0) ** 2
        rms.append(math.sqrt(total / 40))
    assert rms[0] <= 1.25 * rms[1], rms
