"""The isotropic prox of the on-chip solve, which leaves out the square root where a cell surely
shrinks to zero, against the streaming passes.  Both do the same operations on every cell that does
not, so u and phi are equal to the bit wherever the same steps were taken."""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_1808_07284_gb300 as pkg
    assert torch.cuda.is_available()
    return pkg


@pytest.mark.parametrize("nr,nt,tile", [(64, 256, 7), (250, 999, 7), (353, 4001, 10), (640, 5000, 10)])
@pytest.mark.parametrize("scale", [1.0, 1e-13, 1e-15, 1e12])
def test_isotropic_prox_is_the_streaming_one(P, nr, nt, tile, scale):
    """Physical spacings keep most cells at zero and the quiet parts of the records make their flux
    denormal; the unit square opens every cell.  alpha0 sets the threshold: far above the cells' norms,
    about them, and with a square that FP32 cannot hold.  (Not balanced: the means of the two solves come
    from sums of different orders and may round differently.)"""
    obs, pred = synth.gather_pair_hyperbolic(nt=nt, nr=nr, seed=3)
    o, p = (torch.from_numpy(a).cuda() * scale for a in (obs, pred))
    opened = 0
    for dt, dx in ((2e-3, 10.0), (1.0 / (nt - 1), 1.0 / (nr - 1))):
        for alpha0 in (0.0, 1e-6, 1e-24):
            kw = dict(norm=P.EMD_NORM_ISO, balance=P.EMD_BAL_NONE, max_iter=12, alpha0=alpha0, linesearch=0 if alpha0 else 1)
            _, phi, m, a = P.emd(o, p, dt, dx, **kw)
            _, phi0, m0, b = P.emd(o, p, dt, dx, tile=tile, **kw)
            assert a["tile"] == 0 or scale == 1e-15  # (its squares are beneath FP32: handed back)
            assert a["status"] == b["status"] == 0 and a["ls_trials"] == b["ls_trials"]
            assert torch.equal(m, m0) and torch.equal(phi, phi0), (dt, alpha0)
            opened += int((m != 0).any())
    assert opened or scale < 1.0
