"""The benchmark's line names the arithmetic that ran: pruned full passes score candidate
lists in FP32, the tensor cores the dense and the recording ones."""
import sys

import pytest

import bench


@pytest.mark.parametrize("argv,form,dtype", [
    ([], "region", "f32/f64"), (["--precision", "tc_bf16"], "region", "f32/f64"),
    (["--incremental", "2"], "tc_tf32", "tf32/f32/f64"), (["--incremental", "2", "--precision", "fp32"], "region", "f32/f64"), (["--no-prune"], "tc_tf32", "tf32/f32/f64"),
    (["--no-prune", "--precision", "fp32"], "fp32", "f32/f64"),
])
def test_scoring_form(monkeypatch, argv, form, dtype):
    monkeypatch.setattr(sys, "argv", ["bench.py"] + argv)
    args = bench.parse()
    assert bench.scoring_form(args) == form
    assert ("tcgen05" in bench.PRECISION_TEXT[form]) == form.startswith("tc_")
    assert {"tc_tf32": "tf32/f32/f64", "tc_bf16": "bf16/f32/f64"}.get(form, "f32/f64") == dtype
