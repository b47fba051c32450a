"""Byte accounting of the benchmark's kernel records, on CPU with made-up timings."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402
import qadam_inputs as qi  # noqa: E402


class _Handle:
    """What kernel_table asks of a QAdam: sizes and the split between the two worker routes."""

    def __init__(self, D, bits, one_pass, two_pass):
        self.D, self.gcode_bytes, self.wcode_bytes = D, D * bits // 8, D * 2 // 8
        self._model = one_pass, two_pass

    def worker_pass_model(self):
        return self._model


def _profile(**ms):
    names = ("absmax", "quantize", "identity", "server", "broadcast", "worker_fused")
    return {k: (2 * ms.get(k, 0.0), 2 if k in ms else 0) for k in names}


@pytest.mark.parametrize("kg,bits", [(0, 2), (1, 3)])
@pytest.mark.parametrize("one_pass", [0, 3])
def test_sweep_and_the_rows_it_leaves_are_one_pass_over_the_sum_of_their_times(monkeypatch, kg, bits, one_pass):
    # the sweep alone does not write what it leaves to the second kernel, so neither has a rate of its own
    monkeypatch.setattr(bench, "alu_decode_peak", lambda: 1e12)
    w = qi.get_workload("flat20", n=4).with_(kg=kg)
    D, units = 1 << 20, 4 << 20
    q = _Handle(D, bits, one_pass * units // 4, units - one_pass * units // 4)
    t = bench.kernel_table(_profile(absmax=0.8, quantize=0.2, server=0.25), w, "server", q, 0.0, 6500.0)
    assert set(t) == {"sweep", "server"}
    s = t["sweep"]
    assert s["ms_per_launch"] == pytest.approx(1.0) and s["launches"] == 2 and s["share"] == pytest.approx(0.8)
    assert s["algorithmic_bytes"] == (12 + bits / 8) * (units - one_pass * units // 4)
    assert s["achieved_gbs"] == pytest.approx(s["algorithmic_bytes"] / 1e6)


def test_two_full_passes_keep_a_record_each(monkeypatch):
    monkeypatch.setattr(bench, "alu_decode_peak", lambda: 1e12)
    w = qi.get_workload("flat20", n=4)
    q = _Handle(1 << 20, 2, 0, 4 << 20)
    t = bench.kernel_table(_profile(absmax=0.8, quantize=0.2), w, "worker", q, 0.0, 6500.0)
    assert set(t) == {"absmax", "quantize"} and all(k["achieved_gbs"] > 0 for k in t.values())


def test_configurations_the_printed_line_leaves_out_are_counted():
    back = bench.json.loads(bench.printed_line({"value": 1.0, "configs": ["x" * 100] * 100}))
    assert len(back["configs"]) + back["configs_left_out"] == 100 and back["configs_left_out"] > 0
    assert "configs_left_out" not in bench.json.loads(bench.printed_line({"value": 1.0, "configs": ["x"]}))


def test_the_printed_line_is_short_enough_to_be_read_back():
    rec = {"workload": "resnet18_qg_qx_k1", "n_workers": 8, "placement": "worker", "weight_decay": 5e-4,
           "weight_feedback": True, "ms_per_step": 0.0123456789, "step_frac": 0.123456}
    line = {"metric": bench.METRIC, "value": 391295412345.678, "config": {"text": "x" * 800},
            "kernels": {k: {"ms_per_launch": 1.23456789, "frac": 0.123456789} for k in "abcdef"},
            "configs": [bench.config_brief(rec)] * 20}
    short = bench.printed_line(line)
    assert len(short) < bench.LINE_CHARS and len(bench.json.loads(short)["configs"]) == 20
    short = bench.printed_line({**line, "configs": line["configs"] * 5})
    back = bench.json.loads(short)
    assert len(short) < bench.LINE_CHARS and 20 < len(back["configs"]) < 100
    assert back["metric"] == bench.METRIC and abs(back["value"] / line["value"] - 1) < 1e-5
