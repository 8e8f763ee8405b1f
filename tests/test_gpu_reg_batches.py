"""The float register kernels (ks_reg.cuh) in batches large enough to take them (smaller ones take the
items): every covered length of rows and columns, ragged batches whose last tiles are part empty,
explicit steps and loops that freeze, against the items in the persistent kernel, bit for bit; and
the batches on either side of the line."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2007_06427_gb300 import ks_loop as K
from paper_2007_06427_gb300.inputs import spectral_loop

pytestmark = pytest.mark.gpu

# tiles of 1024 points of rows: more than 252 (columns of up to 64, or of 512 points and more) or 380 take
# the kernels
SHAPES = [(32, [32] * 300), (32, [64, 128, 32] * 60), (64, [32, 64, 128, 256] * 14), (64, [512] * 13),
          (128, [128, 32] * 40), (128, [1024, 64, 1024, 64, 1024]), (256, [256, 32] * 6),
          (512, [32, 64, 32] * 7), (512, [1024]),
          (64, [64] * 63), (64, [64] * 64), (64, [128] * 47), (64, [128] * 48), (64, [512] * 7),
          (64, [512] * 8)]  # the line


def descend(nx, ns, path, steps, scheme=K.KS_IMEX, dtau=0.1, tol=0.0):
    L = 22.0 * nx / 64
    seen = {}
    for i, n in enumerate(ns):  # five fields of each length
        if (n, i % 5) not in seen:
            seen[n, i % 5] = spectral_loop(11 + i, nx, L, ns=n, T_range=(20.0, 90.0), decay=(nx / 32.0, 2.0))[:2]
    us, Ts = zip(*[seen[n, i % 5] for i, n in enumerate(ns)])
    u = torch.tensor(np.concatenate([v.ravel() for v in us]), dtype=torch.float32, device="cuda")
    T = torch.tensor(Ts, dtype=torch.float64, device="cuda")
    with K.KSLoop(L, nx, ns, K.KS_FP32, scheme, dtau) as h:
        K.ks_set_option(h.handle, "path", path)
        K.ks_set_state(h.handle, u, T)
        K.ks_step(h.handle, steps, tol)
        band = torch.zeros(2 * K.ks_band_size(h.handle), dtype=torch.float64, device="cuda")
        To = torch.zeros(len(ns), dtype=torch.float64, device="cuda")
        K.ks_get_band(h.handle, band, To)
        steps_o = torch.zeros(len(ns), dtype=torch.int64, device="cuda")
        sq = torch.zeros(len(ns), dtype=torch.float64, device="cuda")
        st = torch.zeros(len(ns), dtype=torch.int32, device="cuda")
        K.ks_get_state(h.handle, u, To, steps_o, sq, st)
    return [x.cpu().numpy() for x in (band, To, u, steps_o, sq, st)]


@pytest.mark.parametrize("nx,ns", SHAPES)
def test_same_bits_as_the_items(nx, ns):
    a, b = (descend(nx, ns, path, 5) for path in (2, 1))
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    assert np.isfinite(a[0]).all() and (a[3] == 5).all()


def test_explicit_steps_and_frozen_loops():
    ns = [64, 128, 32, 256] * 14
    a, ref = (descend(64, ns, path, 7, K.KS_EXPLICIT, 1e-7) for path in (2, 1))
    assert all(np.array_equal(x, y) for x, y in zip(a, ref))
    # a tolerance between the loops' costs freezes some of them at once
    tol = float(np.median(ref[4]))
    a, b = (descend(64, ns, path, 4, K.KS_EXPLICIT, 1e-7, tol) for path in (2, 1))
    assert all(np.array_equal(x, y) for x, y in zip(a, b))
    assert (a[5] == K.KS_CONVERGED).any() and (a[5] == K.KS_RUNNING).any()
