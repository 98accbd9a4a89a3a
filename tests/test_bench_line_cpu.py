"""The bench's line on standard output stays short whatever the workloads beside the headline one
record, and keeps the keys that its readers use."""
import json

import bench


def _full_record():
    arm = dict(cycles=15, cycle_ms=3.5708182879856656, eps_T=0.3491818194105757,
               mse_per_cycle=[0.0009739572997204959] * 15)
    baseline = dict(value=0.1721454465942213, unit="GLUPS", cores=16, kind="oracle",
                    sample="FP64 C oracle, OpenMP rows on 16 host threads: 9219 LBM steps of one 512x256 porous "
                           "trajectory (seed 0) in 7.0 s", single_thread=dict(value=0.0123456789, unit="GLUPS",
                                                                             cores=1, sample="1234 steps in 7.0 s"),
                    fno_oracle=dict(seconds=7.123456789, sample="x" * 120))
    return dict(
        metric=bench.METRIC, value=137.50516220760298, unit="GLUPS", n_gpus=1, steps=20, warmup=5,
        ms_per_step=1220.1153564453125, higher_is_better=True, scaling="weak", vs_baseline=None, dtype="f32",
        data="synthetic", config=bench.bench_config(64, [0.601123, 0.790456], 20000, 1),
        roofline=dict(bound="hbm", achieved=5273.647914028307, peak=6787.2, unit="GB/s", frac=0.7755364579453393,
                      peak_kind="measured", kernel="k_sweep", bytes_per_launch=605028352.0, steps_per_launch=2,
                      check_step_tile_shape=dict(rows_per_tile=5, stages=2, ctas_per_sm=4),
                      launch_ms=0.11472672462463379, traffic=553958144.0,
                      traffic_unit="bytes per launch (ncu dram read + write)"),
        reinit_kernel=dict(kernel="k_reinit", neq_mode=1, launch_ms=0.12913440465927123, bytes_per_launch=469762048,
                           achieved_gbs=3637.7760770996315, frac_of_measured_hbm=0.5349670701617105),
        time_to_steady_summary=dict(tol=1e-5, trajectories=20, fno_init_s=0.7995745849609375, fno_init_converged=True,
                                    plain_init_s=3.37962158203125, plain_init_converged=False, step_cap=150000),
        solve=dict(lbm_steps=20000, converged=False, max_residual=0.00045007553452699166),
        time_to_steady=dict(seconds=[0.5] * 200), tolerance_ladder=dict(rows=[0.123456789] * 600),
        lbm_sweep=[dict(nx=4096, glups=141.1209399153309)] * 3, launch_bound=dict(a=[1.0] * 100),
        hybrid_training=dict(ms_per_step=23.246829223632812), double_shear=dict(arms={"1:1": arm, "1:2": arm, "1:3": arm,
                                                                                      "fno_only": dict(cycle_ms=0.9)}),
        fno_throughput=dict(ms_per_forward=0.5490799903869629), unsteady_hybrid=dict(cycle_ms_steady=9.975287437438965),
        autotune_ms=[0.09971839934587479] * 6, gpu_launches=212540,
        clocks=dict(sm_mhz=2070.0, sm_max_mhz=2070.0, reasons=[], samples=1200),
        e2e=dict(value=136.52875748669527, unit="GLUPS", h2d_bytes_per_step=1048576, d2h_bytes_per_step=100663296),
        cpu_baseline=baseline)


def test_line_is_short_and_complete():
    record = _full_record()
    line, details = bench.split_line(record)
    text = json.dumps(line)
    assert len(text) <= bench.LINE_MAX < len(json.dumps(record)), len(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "roofline", "clocks", "e2e", "gpu_launches", "cpu_baseline"):
        assert key in line, key
    assert abs(line["value"] / record["value"] - 1) < 1e-6 and line["e2e"]["d2h_bytes_per_step"] == 100663296
    assert set(details) == set(bench.DETAIL_KEYS) and details["tolerance_ladder"] == record["tolerance_ladder"]
    assert line["other"]["shear_eps_T"] == {"1:1": 0.3491818, "1:2": 0.3491818, "1:3": 0.3491818}


def test_line_without_the_other_workloads():
    record = {k: v for k, v in _full_record().items() if k not in bench.DETAIL_KEYS}
    record.update({k: None for k in bench.DETAIL_KEYS})
    line, _ = bench.split_line(record)
    assert set(line["other"].values()) == {None} and len(json.dumps(line)) <= bench.LINE_MAX
