"""The benchmark's result line: short enough for a reader that keeps the end of the
output, and no conversion on the tensor cores graded against the CUDA-core probe.
"""
import json

import bench
import oracle


def test_autotuner_report_is_the_choice_and_a_count():
    best = (1, 8, 2, 15, 8, 7, 0, 0, 0, 0.1940000057220459)
    rep = bench.tune_report(best, [best] * 300)
    assert rep == dict(bench.shape_dict(best), shapes_timed=300)
    assert len(json.dumps(bench.short(rep))) < 200


def test_short_keeps_six_digits_and_the_rest():
    o = {"a": 1.23456789e-9, "b": [3846.887722860725, 7, None, "x", True], "c": {"d": 12345678}}
    assert bench.short(o) == {"a": 1.23457e-9, "b": [3846.89, 7, None, "x", True], "c": {"d": 12345678}}


def test_tensor_conversions_follow_the_primes():
    assert all(bench.tensor_conversions(oracle.preset(n).ext) for n in ("n15", "n16", "n17"))
    assert not bench.tensor_conversions(oracle.preset("n12").ext)
    assert not bench.tensor_conversions(oracle.make_params(12, 4, 2, 2, 55, 56).ext)
