"""The bench's FP64 roofline is of the FP64 unit's instructions (the formulas' FLOPs run on the integer units too and
would pass the unit's rate)."""
import importlib.util
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _bench():
    spec = importlib.util.spec_from_file_location("bench_roofline", os.path.join(ROOT, "bench.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    return b


def test_fp64_rate_counts_instructions_of_the_current_capture():
    b = _bench()
    rec = b.capture_record("predictor_faces", 3, "nodal", False)
    assert rec is not None
    zones, seconds = 256 ** 3, 0.042
    got = b.fp64_instruction_rate("predictor_faces", 3, "nodal", zones, seconds)
    assert got == rec["fp64_instructions_per_zone"] * zones / seconds / 1e12
    # two a clock and SM, 152 SMs, is the most the unit executes: the measured launch stays below it
    assert 0.3 < got / (b.alu_peak_tflops(False, 2070.0) / 2) < 1.0
    # the formulas' FLOPs do not: they pass an FMA's two FLOPs for each of those instructions
    assert b.flops_per_zone(3, "nodal", "hll", False, tiled=False)["predictor_faces"] > 2 * rec["fp64_instructions_per_zone"]


def test_no_rate_without_a_capture_of_the_configuration():
    b = _bench()
    assert b.fp64_instruction_rate("predictor_faces", 4, "modal", 1000, 1e-3) is None
    assert b.fp64_instruction_rate("weno_reconstruction", 3, "nodal", 1000, 1e-3) is None
