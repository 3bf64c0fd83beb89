"""The benchmark's printed line: short, and with every key of its contract (no GPU needed)."""
import json

import bench
import workloads


def record(workload):
    w = workloads.by_name(workload)
    num = 0.012345678901234567
    roof = dict(kernel="zta_pair_kernel", bound="tensor", achieved=1234.567890123, peak=1647.6, unit="TFLOP/s", frac=num, traffic=None,
                kernel_ms=num, share_of_step=num, peak_source="measured", note="n" * 400, step=dict(note="n" * 400))
    configs = {k: dict(workload="x" * 40, us=123.45, ex_s=1e6 / 7, bound="hbm", roof_us=12.34, frac=0.1234, frac_sustained=0.1234)
               for k in ("cfg1", "cfg2", "cfg2_bf16", "cfg3_f32", "cfg3_bf16", "cfg4")}
    configs["cfg5"] = {f"{k},2048,4096,1024": [123.4, 0.123] for k in range(24)}
    return dict(metric=bench.METRIC, value=1e6 / 7, unit=bench.UNIT, n_gpus=1, steps=50, warmup=10, ms_per_step=num,
                higher_is_better=True, scaling="weak", vs_baseline=None, dtype=w.dtype, data="synthetic",
                config=bench.workload_config(w, 1), gpu_launches=4 * 50,
                clocks=dict(sm_mhz=1965.0, sm_max_mhz=1965.0, reasons=["sw_power_cap"], samples=30), roofline=roof,
                step_roofline_frac=num, warm_l2_ms_per_step=num, eager_ms_per_step=num, one_stream_graph_ms_per_step=num,
                launch="l" * 130, breakdown_us={f"k{i}": num for i in range(20)},
                e2e=dict(value=num, unit=bench.UNIT, h2d_bytes_per_step=10 ** 9, d2h_bytes_per_step=10 ** 7, ms_per_step=num,
                         serial_ms_per_step=num, note="n" * 200),
                cpu_baseline=dict(value=num, unit=bench.UNIT, cores=1, kind="oracle", sample="s" * 140),
                workloads={f"w{i}": dict(note="n" * 1000) for i in range(12)}, configs=configs)


def test_printed_line_is_short_and_complete(capsys):
    for workload in ("cfg1", "cfg2", "cfg2_bf16", "cfg3_f32", "cfg3_bf16", "cfg4"):
        r = record(workload)
        bench.emit(r)
        out, err = capsys.readouterr()
        assert out.count("\n") == 1 and len(out) <= bench.HEADLINE_MAX + 1
        line = json.loads(out)
        for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
                  "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
            assert k in line, k
            if k not in ("e2e", "roofline"):
                assert line[k] == r[k]
        assert line["configs"]["cfg4"] == [123.45, 0.1234] and {"value", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(line["e2e"])
        assert json.loads(err) == json.loads(json.dumps(r))
