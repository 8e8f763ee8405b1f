"""The float phases with the transforms in registers (ks_reg.cuh) against the items they stand in
for: every covered length of rows and columns, ragged batches whose last tiles are part empty, the
subspace and the uncovered lengths (which take the items), frozen loops.  The arithmetic is the
same, so the results are compared bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2007_06427_gb300 import ks_loop as K
from paper_2007_06427_gb300.inputs import spectral_loop

pytestmark = pytest.mark.gpu

SHAPES = [(32, [32]), (32, [64, 32, 128]), (64, [32, 64, 128, 256, 64]), (64, [512]), (128, [128, 32]),
          (128, [1024, 64, 1024]), (256, [256, 32]), (512, [32, 64, 32]), (512, [1024]),
          (64, [16, 64]), (16, [64]), (1024, [32])]    # the last three: items


def descend(nx, ns, path, steps, L, xi=0, scheme=K.KS_IMEX, dtau=0.1, tol=0.0):
    us, Ts = [], []
    for i, n in enumerate(ns):
        u, T, _ = spectral_loop(11 + i, nx, L, ns=n, T_range=(20.0, 90.0), decay=(nx / 32.0, 2.0),
                                symmetric=bool(xi))
        us.append(u.ravel())
        Ts.append(T)
    u = torch.tensor(np.concatenate(us), dtype=torch.float32, device="cuda")
    T = torch.tensor(Ts, dtype=torch.float64, device="cuda")
    with K.KSLoop(L, nx, ns, K.KS_FP32, scheme, dtau) as h:
        K.ks_set_option(h.handle, "path", path)
        K.ks_set_option(h.handle, "symmetry", xi)
        K.ks_set_state(h.handle, u, T)
        K.ks_step(h.handle, steps, tol)
        band = torch.zeros(2 * K.ks_band_size(h.handle), dtype=torch.float64, device="cuda")
        To = torch.zeros(len(ns), dtype=torch.float64, device="cuda")
        K.ks_get_band(h.handle, band, To)
        uo = torch.empty_like(u)
        steps_o = torch.zeros(len(ns), dtype=torch.int64, device="cuda")
        sq = torch.zeros(len(ns), dtype=torch.float64, device="cuda")
        st = torch.zeros(len(ns), dtype=torch.int32, device="cuda")
        K.ks_get_state(h.handle, uo, To, steps_o, sq, st)
    return [x.cpu().numpy() for x in (band, To, uo, steps_o, sq, st)]


@pytest.mark.parametrize("nx,ns", SHAPES)
@pytest.mark.parametrize("xi", [0, 1])
def test_same_bits_as_the_items(nx, ns, xi):
    a = descend(nx, ns, 2, 5, 22.0 * nx / 64, xi)
    b = descend(nx, ns, 1, 5, 22.0 * nx / 64, xi)    # the persistent kernel runs the items
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    assert np.isfinite(a[0]).all() and (a[3] == 5).all()


def test_explicit_steps_and_frozen_loops():
    for path in (1, 2):
        r = descend(64, [64, 128, 64], path, 7, 22.0, scheme=K.KS_EXPLICIT, dtau=1e-7)
        if path == 1:
            ref = r
    assert all(np.array_equal(x, y) for x, y in zip(r, ref))
    # a tolerance between the loops' costs freezes some of them at once
    sq = np.sort(ref[4])
    tol = 0.5 * (sq[0] + sq[1])
    a, b = (descend(64, [64, 128, 64], p, 4, 22.0, scheme=K.KS_EXPLICIT, dtau=1e-7, tol=float(tol))
            for p in (1, 2))
    assert all(np.array_equal(x, y) for x, y in zip(a, b))
    assert (a[5] == K.KS_CONVERGED).any() and (a[5] == K.KS_RUNNING).any()


@pytest.mark.parametrize("nx,ns", [(64, [32] * 40 + [64] * 30 + [128, 256] * 20 + [512]), (64, [64] * 120),
                                   (32, [128, 256] * 60), (128, [1024] * 5 + [32] * 90)])
def test_column_groups_have_the_items_bits(nx, ns):
    """The double column phases by groups of columns (large batches) against the items."""
    outs = []
    L = 22.0 * nx / 64
    us, Ts = zip(*[spectral_loop(i, nx, L, ns=n, T_range=(20.0, 90.0))[:2] for i, n in enumerate(ns)])
    for path in (2, 1):
        u = torch.tensor(np.concatenate([v.ravel() for v in us]), device="cuda")
        T = torch.tensor(Ts, dtype=torch.float64, device="cuda")
        sq = torch.zeros(len(ns), dtype=torch.float64, device="cuda")
        with K.KSLoop(L, nx, ns, K.KS_FP64, K.KS_IMEX, 0.1) as h:
            K.ks_set_option(h.handle, "path", path)
            K.ks_set_state(h.handle, u, T)
            K.ks_step(h.handle, 3, 0.0)
            K.ks_get_state(h.handle, u, T, None, sq)
        outs.append([x.cpu().numpy() for x in (u, T, sq)])
    for x, y in zip(*outs):
        assert np.isfinite(x).all() and np.array_equal(x, y)
