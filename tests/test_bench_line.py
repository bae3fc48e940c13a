"""The benchmark's one JSON line: short enough to be read back from the end of the output, with every key of its
contract as measured, whatever further measurements ran."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_line_is_short_and_whole():
    sys.path.insert(0, ROOT)
    import bench
    line = {k: None for k in bench.LINE_KEYS}
    line.update(metric=bench.METRIC, value=1218062411096.8188, unit=bench.UNIT, n_gpus=1, steps=20, warmup=5,
                ms_per_step=6.567807960510254, higher_is_better=True, scaling="weak", gpu_launches=80,
                e2e={"value": 1143315514379.9373, "unit": bench.UNIT, "h2d_bytes_per_step": 128000000,
                     "d2h_bytes_per_step": 96000088},
                clocks={"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, sweep=[{"x" * 20: 1.0 / 3} for _ in range(600)],
                slab={"ms_per_step": 0.07325120121240616},
                npt_one_replica={"by_N": {str(10 ** k): {"fp32_ms_per_step": 0.1, "fp64_ms_per_step": 0.2} for k in range(60)}})
    out = bench.short_line(line)
    text = json.dumps(out)
    assert len(text) <= bench.LINE_MAX and "\n" not in text
    for k in bench.LINE_KEYS:
        assert out[k] == line[k]
    assert out["also"]["slab_ms"] == 0.0732512 and "sweep" not in out
