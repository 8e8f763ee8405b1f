"""The launch form of a resumed handle, with a library that only keeps the knobs (no GPU): a file that
records "path_auto" restores it, one from before that knob leaves the rule in force unless its path
differs from the value a handle is created with."""
import numpy as np
import pytest

from paper_2007_06427_gb300 import checkpoint


class Loop:
    def __init__(self, L, nx, ns, mode, scheme, dtau, **kw):
        self.L, self.nx, self.ns, self.mode, self.scheme, self.dtau = L, nx, ns, mode, scheme, dtau
        self.batch = len(ns)
        # as the library creates a double 64 x 256 loop: path 2 until set, and the rule in force
        self.handle = {"path_f64": 2, "path_f32": 0, "path_auto": 3}

    def close(self):
        pass


def set_option(handle, key, value):
    if key == "path_f64":
        handle["path_auto"] &= ~1
    if key == "path_f32":
        handle["path_auto"] &= ~2
    handle[key] = value


@pytest.mark.parametrize("knobs,auto,path", [
    (dict(path_f64=2, path_f32=0), 3, 2),                       # an old file of an untouched handle
    (dict(path_f64=0, path_f32=0), 2, 0),                       # an old file whose double path was set
    (dict(path_f64=2, path_f32=0, path_auto=3), 3, 2),
    (dict(path_f64=2, path_f32=0, path_auto=0), 0, 2),          # set to the value at create
    (dict(path_f64=1, path_f32=1, path_auto=0), 0, 1)])
def test_form_of_a_resumed_handle(tmp_path, monkeypatch, knobs, auto, path):
    monkeypatch.setattr(checkpoint.K, "KSLoop", Loop)
    monkeypatch.setattr(checkpoint.K, "ks_band_size", lambda h: 4)
    monkeypatch.setattr(checkpoint.K, "ks_set_band", lambda *a: None)
    monkeypatch.setattr(checkpoint.K, "ks_set_option", set_option)
    monkeypatch.setattr(checkpoint.K, "ks_get_option", lambda h, k: h[k])
    f = tmp_path / "c.npz"
    np.savez(f, L=22.0, nx=64, ns=np.array([256]), mode=0, scheme=1, dtau=0.1, tol=1e-10, switch_tol=0.0,
             band=np.zeros(8), T=np.zeros(1), prec=np.zeros(1, np.int32), steps=np.zeros(1, np.int64),
             status=np.zeros(1, np.int32), version=checkpoint.VERSION,
             **{f"knob_{k}": v for k, v in knobs.items()})
    loop = checkpoint.resume(str(f))
    assert (loop.handle["path_auto"], loop.handle["path_f64"]) == (auto, path)
