"""r and G of the double path against a long double evaluation (dense transforms): at most half the error of
a double evaluation of the same sums, the oracle's.  The margin is the transforms' (64-bit fixed point,
and the residual from the spectrum of u^2): a double transform of u u_x is as far off as the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ks_oracle as ko
from paper_2007_06427_gb300 import ks_loop as K
from paper_2007_06427_gb300.inputs import spectral_loop

pytestmark = pytest.mark.gpu

PI = np.longdouble("3.14159265358979323846264338327950288")


def dense(n):
    t = (np.outer(np.arange(n), np.arange(n)) % n).astype(np.longdouble) * (2 * PI / n)
    return np.cos(t) + 1j * np.sin(t)


def in_long_double(u, T, L):
    ns, nx = u.shape
    L, T = np.longdouble(L), np.longdouble(T)
    ex, es = dense(nx), dense(ns)
    j, k = (np.fft.fftfreq(n, 1.0 / n).astype(int) for n in (nx, ns))
    keep = (np.abs(k)[:, None] <= ns // 3) & (np.abs(j)[None, :] <= nx // 3)
    q, om = (2 * PI * j / L)[None, :], (2 * PI * k / T)[:, None]

    def hat(f):
        return es.conj() @ f.astype(np.clongdouble) @ ex.conj() / (nx * ns) * keep

    def grid(h):
        return (es @ h @ ex).real

    uh = hat(u.astype(np.longdouble))
    ug = grid(uh)
    rh = (q**2 - q**4 - 1j * om) * uh - hat(ug * grid(1j * q * uh))
    return grid(rh), grid((q**2 - q**4 + 1j * om) * rh + hat(ug * grid(1j * q * rh)))


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 60, reason="no long double")
@pytest.mark.parametrize("nx,ns,L,decay", [(32, 32, 22.0, 2.0), (64, 64, 22.0, 2.0), (128, 64, 44.0, 4.0),
                                           (64, 128, 39.0, 2.0)])
def test_no_further_than_half_a_double_evaluation(nx, ns, L, decay):
    u, T, _ = spectral_loop(1, nx, L, ns=ns, T_range=(20.0, 80.0), decay=(decay, 2.0))
    ud = torch.tensor(u.ravel(), device="cuda")
    Td = torch.tensor([T], dtype=torch.float64, device="cuda")
    r, G, s = torch.empty_like(ud), torch.empty_like(ud), torch.empty_like(Td)
    with K.KSLoop(L, nx, [ns], K.KS_FP64) as h:
        K.ks_residual(h.handle, ud, Td, r, s)
        K.ks_adjoint_grad(h.handle, ud, Td, G, s)
    ref = ko.adjoint_grad(u, T, L)
    host = ko.grid(nx, ns, L).real_grid(ref["rh"]), ref["G"]
    for exact, gpu, double in zip(in_long_double(u, T, L), (r, G), host):
        def off(x):
            return float(np.linalg.norm((x - exact).astype(np.float64)))
        assert off(gpu.cpu().numpy().reshape(ns, nx)) <= 0.5 * off(double)
