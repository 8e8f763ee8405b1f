"""The launch form of a handle whose "path" knob is not set: which one the rule takes on either side of
its lines, that setting the knob or "path_auto" wins, and that the results have the other forms' bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2007_06427_gb300 import ks_loop as K
from paper_2007_06427_gb300.inputs import spectral_loop

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,nx,ns,form", [
    (K.KS_FP64, 64, [128], 0), (K.KS_FP64, 64, [256], 0), (K.KS_FP64, 64, [64] * 16, 0),
    (K.KS_FP64, 64, [128] * 8, 0), (K.KS_FP64, 128, [256], 2), (K.KS_FP64, 32, [64] * 256, 2),
    (K.KS_FP64, 64, [32, 64, 128, 256] * 16, 2), (K.KS_FP32, 64, [64] * 256, 2),
    (K.KS_FP32, 128, [256], 0), (K.KS_FP32, 256, [256], 2), (K.KS_FP32, 256, [32] * 64, 2),
    (K.KS_FP32, 64, [256] * 4, 0)])
def test_rule_and_bits(mode, nx, ns, form):
    f32 = mode == K.KS_FP32
    L = 22.0 * nx / 64
    us, Ts = zip(*[spectral_loop(3 + i, nx, L, ns=n, T_range=(20.0, 90.0), decay=(nx / 32.0, 2.0))[:2]
                   for i, n in enumerate(ns)])
    outs = []
    for path in (None, 2 - form):
        u = torch.tensor(np.concatenate([v.ravel() for v in us]), device="cuda",
                         dtype=torch.float32 if f32 else torch.float64)
        T = torch.tensor(Ts, dtype=torch.float64, device="cuda")
        with K.KSLoop(L, nx, ns, mode, K.KS_IMEX, 0.1) as h:
            key = "form_f32" if f32 else "form_f64"
            assert K.ks_get_option(h.handle, "path_auto") == 3
            assert K.ks_get_option(h.handle, key) == form
            if path is not None:
                K.ks_set_option(h.handle, "path", path)
                assert K.ks_get_option(h.handle, "path_auto") == 0
                assert K.ks_get_option(h.handle, key) == path
            K.ks_set_state(h.handle, u, T)
            K.ks_step(h.handle, 3, 0.0)
            sq = torch.zeros(len(ns), dtype=torch.float64, device="cuda")
            K.ks_get_state(h.handle, u, T, None, sq)
            K.ks_set_option(h.handle, "path_auto", 3)
            assert K.ks_get_option(h.handle, key) == form
        outs.append([x.cpu().numpy() for x in (u, T, sq)])
    for a, b in zip(*outs):
        assert np.isfinite(a).all() and np.array_equal(a, b)
