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


def relative(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("nx,nss", [(32, [32, 16]), (64, [128, 64, 8]), (256, [256]), (128, [512, 32]), (32, [1024])])
@pytest.mark.parametrize("amps", [(1e-33,), (1e-40,), (1e33,), (1.0, 1e-33, 1e33)])
def test_residual_and_gradient_outside_the_float_range(nx, nss, amps):
    """Amplitudes where every scale, or that of a neighbouring loop, comes from the exponents, at lengths on
    both sides of 128 (where the scale has a pass of its own), against the oracle: 1e-12 of each
    loop's norm, as for ordinary loops."""
    from oracle import ks_oracle as ko
    L = 22.0 * max(1.0, nx / 64)
    nss = nss * len(amps)
    us, Ts = loops(nx, nss, L, amps, decay=(max(2.0, (nx // 3) / 10.0), 2.0))
    u = torch.tensor(np.concatenate([a.ravel() for a in us]), device="cuda")
    T = torch.tensor(Ts, dtype=torch.float64, device="cuda")
    r, G = torch.empty_like(u), torch.empty_like(u)
    J, dJ = torch.empty_like(T), torch.empty_like(T)
    with K.KSLoop(L, nx, nss, K.KS_FP64) as h:
        K.ks_residual(h.handle, u, T, r, J)
        K.ks_adjoint_grad(h.handle, u, T, G, dJ)
    at = 0
    for b, n in enumerate(nss):
        ref = ko.adjoint_grad(us[b], Ts[b], L)
        r_ref = ko.grid(nx, n, L).real_grid(ref["rh"])
        cut = slice(at, at + n * nx)
        at += n * nx
        assert relative(r.cpu().numpy()[cut], r_ref.ravel()) < 1e-12
        assert relative(G.cpu().numpy()[cut], ref["G"].ravel()) < 1e-12
        assert abs(J[b].item() - ref["J"]) <= 1e-12 * ref["J"]
