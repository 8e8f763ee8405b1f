"""The launch form of float handles whose "path" knob is not set on either side of the rule's lines for long
transforms, small batches and the subspace, with the same bits as the other form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2007_06427_gb300 import ks_loop as K
from paper_2007_06427_gb300.inputs import spectral_loop

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ns,xi,form", [
    (32, [1024], 0, 2), (64, [512], 0, 2), (64, [512] * 18, 0, 2), (32, [512], 0, 0), (1024, [32], 0, 2),
    (256, [128] * 8, 0, 2), (256, [128] * 4, 0, 0), (64, [32, 64, 128, 256] * 8, 0, 0),
    (32, [1024], 1, 2), (64, [512], 1, 0), (128, [32] * 300, 1, 0), (128, [64] * 120, 1, 2)])
def test_rule_and_bits(nx, ns, xi, form):
    L = 22.0 * nx / 64
    us, Ts = zip(*[spectral_loop(3 + i % 7, nx, L, ns=n, T_range=(20.0, 90.0), decay=(nx / 32.0, 2.0),
                                 symmetric=bool(xi))[:2] for i, n in enumerate(ns)])
    outs = []
    for path in (None, 2 - form):
        u = torch.tensor(np.concatenate([v.ravel() for v in us]), device="cuda", dtype=torch.float32)
        T = torch.tensor(Ts, dtype=torch.float64, device="cuda")
        with K.KSLoop(L, nx, ns, K.KS_FP32, K.KS_IMEX, 0.1) as h:
            K.ks_set_option(h.handle, "symmetry", xi)
            assert K.ks_get_option(h.handle, "form_f32") == form
            if path is not None:
                K.ks_set_option(h.handle, "path", path)
            K.ks_set_state(h.handle, u, T)
            K.ks_step(h.handle, 3, 0.0)
            sq = torch.zeros(len(ns), dtype=torch.float64, device="cuda")
            K.ks_get_state(h.handle, u, T, None, sq)
        outs.append([x.cpu().numpy() for x in (u, T, sq)])
    for a, b in zip(*outs):
        assert np.isfinite(a).all() and np.array_equal(a, b)
