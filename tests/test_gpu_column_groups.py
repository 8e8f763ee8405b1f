"""The double column phases by groups of columns (batches of at least 304 groups) in what the IMEX steps of
running loops do not reach: explicit steps, loops that freeze while others run, loops of a mixed batch
that come to double one by one, steep spectra whose columns differ by tens of orders of magnitude
inside a group.  Against the items in the persistent kernel, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2007_06427_gb300 import ks_loop as K
from paper_2007_06427_gb300.inputs import spectral_loop

pytestmark = pytest.mark.gpu

NX, L = 64, 22.0
NS = [32, 64, 128, 256, 64, 32, 128] * 12   # 84 loops, more than 400 groups


def batch(decay=(2.0, 2.0), amps=(1.0,)):
    us, Ts = zip(*[spectral_loop(i % 9, NX, L, ns=n, T_range=(20.0, 90.0), decay=decay)[:2]
                   for i, n in enumerate(NS)])
    u = np.concatenate([v.ravel() * amps[i % len(amps)] for i, v in enumerate(us)])
    return torch.tensor(u, device="cuda"), torch.tensor(Ts, dtype=torch.float64, device="cuda")


def stepped(path, scheme, dtau, steps, tol=0.0, **kw):
    u, T = batch(**kw)
    sq = torch.zeros(len(NS), dtype=torch.float64, device="cuda")
    st = torch.zeros(len(NS), dtype=torch.int32, device="cuda")
    n = torch.zeros(len(NS), dtype=torch.int64, device="cuda")
    with K.KSLoop(L, NX, NS, K.KS_FP64, scheme, dtau) as h:
        K.ks_set_option(h.handle, "path", path)
        K.ks_set_state(h.handle, u, T)
        K.ks_step(h.handle, steps, tol)
        band = torch.zeros(2 * K.ks_band_size(h.handle), dtype=torch.float64, device="cuda")
        K.ks_get_band(h.handle, band, T)
        K.ks_get_state(h.handle, u, T, n, sq, st)
    return [x.cpu().numpy() for x in (band, T, u, n, sq, st)]


def same(a, b):
    assert all(np.isfinite(x).all() for x in a)
    assert all(np.array_equal(x, y) for x, y in zip(a, b))


def test_explicit_steps():
    same(*(stepped(p, K.KS_EXPLICIT, 1e-7, 5) for p in (2, 1)))


def test_loops_that_freeze():
    ref = stepped(1, K.KS_IMEX, 0.1, 6)
    # the median cost after six steps: half the loops freeze on the way there, the others run on
    tol = float(np.median(ref[4]))
    a, b = (stepped(p, K.KS_IMEX, 0.1, 6, tol) for p in (2, 1))
    same(a, b)
    assert len(set(a[3].tolist())) > 1 and (a[5] == K.KS_CONVERGED).any() and (a[5] == K.KS_RUNNING).any()


def test_steep_spectra():
    """Columns fall by e^-4 per mode and loops by 1e-20: groups hold transforms on both sides of the line
    where the scale comes from the exponents."""
    same(*(stepped(p, K.KS_IMEX, 0.1, 4, decay=(0.25, 1.0), amps=(1.0, 1e-10, 1e-20)) for p in (2, 1)))


def test_mixed_batch():
    out = []
    for path in (2, 1):
        u, T = batch()
        steps = torch.zeros(len(NS), dtype=torch.int64, device="cuda")
        sq = torch.zeros(len(NS), dtype=torch.float64, device="cuda")
        st = torch.zeros(len(NS), dtype=torch.int32, device="cuda")
        with K.KSLoop(L, NX, NS, K.KS_MIXED, K.KS_IMEX, 0.1, switch_tol=3.0, chunk=10) as h:
            K.ks_set_option(h.handle, "path", path)
            K.ks_descend(h.handle, u, T, 60, 0.5, steps, sq, st)
        out.append([x.cpu().numpy() for x in (u, T, steps, sq, st)])
    same(*out)
