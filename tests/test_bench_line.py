"""The benchmark's standard output is one short JSON line (no GPU needed)."""
import json

import bench


def test_headline_alone_on_standard_output(capsys):
    line = {"metric": bench.METRIC, "value": 1.5, "unit": bench.UNIT}
    extra = {"serving": {"levels": [{"p50_ms": 0.1 * i} for i in range(2000)]}, "sampler": {"n": 1}}
    bench.emit(line, extra)
    got = capsys.readouterr()
    assert got.out.count("\n") == 1 and json.loads(got.out) == line
    assert {k for row in got.err.splitlines() for k in json.loads(row)} == set(extra)


def test_work_counts_split_by_pipe():
    """Every multiply-add of a result with its estimate runs on one of the two."""
    for n in range(2, 31, 2):
        total = bench.fixed_point_flops(n) + bench.fp64_flops(n)
        assert total == 8 * (bench.matching_macs(n) + bench.term_macs(n))
        assert (bench.fixed_point_flops(n) > 0) == (n >= 12)
    assert abs(bench.fixed_point_peak_tflops() / (152 * 4 * 32 / 28 * 8 * 2.07e-3) - 1) < 1e-12
