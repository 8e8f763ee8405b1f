"""The launch forms on loops of small amplitude: their products u^2 and u r_x fall through the line
(2^-100 of a transform's sum of moduli) where the fixed-point double transforms take their scale
from the exponents instead of a float sum, column by column.  The forms still compute the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2007_06427_gb300 import ks_loop as K
from paper_2007_06427_gb300.inputs import spectral_loop

pytestmark = pytest.mark.gpu


def loops(nx, nss, L, amps, xi=0, decay=(2.0, 2.0)):
    us, Ts = [], []
    for i, n in enumerate(nss):
        u, T, _ = spectral_loop(5 + i, nx, L, ns=n, T_range=(20.0, 80.0), decay=decay, symmetric=bool(xi))
        us.append(u * amps[i % len(amps)])
        Ts.append(T)
    return us, Ts


def stepped(us, Ts, nx, nss, L, path, xi, steps=4):
    u = torch.tensor(np.concatenate([a.ravel() for a in us]), device="cuda")
    T = torch.tensor(Ts, dtype=torch.float64, device="cuda")
    sq = torch.zeros(len(nss), dtype=torch.float64, device="cuda")
    with K.KSLoop(L, nx, nss, K.KS_FP64, K.KS_IMEX, 0.1) as h:
        K.ks_set_option(h.handle, "path", path)
        K.ks_set_option(h.handle, "symmetry", xi)
        K.ks_set_state(h.handle, u, T)
        K.ks_step(h.handle, steps, 0.0)
        band = torch.zeros(2 * K.ks_band_size(h.handle), dtype=torch.float64, device="cuda")
        K.ks_get_band(h.handle, band, T)
        K.ks_get_state(h.handle, u, T, None, sq)
    return [x.cpu().numpy() for x in (band, T, u, sq)]


@pytest.mark.parametrize("xi", [0, 1])
@pytest.mark.parametrize("nx,nss", [(64, [128]), (64, [64] * 7), (32, [32, 256, 16]), (128, [512, 64]),
                                    (64, [128] * 120)])
@pytest.mark.parametrize("exponent", [-14, -15, -16, -17])
def test_forms_agree_across_the_line(exponent, nx, nss, xi):
    L = 22.0 * max(1.0, nx / 64)
    us, Ts = loops(nx, nss, L, [m * 10.0**exponent for m in (1.0, 2.5, 6.0)], xi, (nx / 32.0, 2.0))
    ref = stepped(us, Ts, nx, nss, L, 2, xi)
    assert all(np.isfinite(x).all() for x in ref)
    for path in (0, 1):
        for x, y in zip(stepped(us, Ts, nx, nss, L, path, xi), ref):
            assert np.array_equal(x, y)
