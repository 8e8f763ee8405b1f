"""The per-SM fraction of the bench's roofline follows the kernel that ran, not the "path" knob: a handle
whose knob says four launches can run the cluster kernel by the launch-form rule, and the reverse."""
import pytest

torch = pytest.importorskip("torch")

import bench


class H:
    handle = None


class Props:
    multi_processor_count = 152


@pytest.mark.parametrize("path,kernel,used", [(2, "cluster_f64", 16), (0, "cluster_f64", 16), (0, "rows_adj_f64", None),
                                              (2, "cols_resid_f64", None), (0, "persist_f64", None)])
def test_sms_of_the_kernel_that_ran(monkeypatch, path, kernel, used):
    class FakeK:
        KS_FP32 = 1

        @staticmethod
        def ks_get_option(handle, key):
            return {"path": path, "cluster_f64": 16}[key]

    monkeypatch.setattr(torch.cuda, "get_device_properties", lambda dev: Props())
    r = bench.annotate_sms({"kernel": kernel, "frac": 0.01}, FakeK, H, 0, 1, None)
    assert r.get("sms_used") == used
    if used:
        assert abs(r["frac_of_sms_used"] - 0.01 * 152 / used) < 1e-15
