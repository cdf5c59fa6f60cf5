"""The benchmark's stdout line: the contract's entries in a line short enough to be
kept whole by whoever logs only the end of the output."""
import json

import bench


def _record():
    trial = dict(n_group=16, n_leaf=16, pair_targets=16, pair_warps=4, pair_unroll=4, ms_per_step=2.4368690047)
    roof = dict(kernel="nlist_kernel", bound="alu", achieved=4.573, peak=80.01, unit="TFLOP/s", frac=0.0572,
                peak_basis="measured " * 30, stages={k: dict(trial) for k in ("lists", "density", "force")})
    stage = {k: 0.3628 for k in ("tree", "density", "force", "reduce", "leapfrog", "prep", "lists", "gravity")}
    leg = dict(workload="w" * 90, value=733620229.1370077, unit="particle-updates/s", roofline=roof,
               autotune=dict(trial, trials=[trial] * 20), stage_ms=stage)
    clocks = dict(sm_mhz=2070.0, sm_max_mhz=2070.0, reasons=["sw_power_cap"], samples=24, after_region=dict(stage))
    return dict(
        metric=bench.METRIC, value=913043146.2817698, unit=bench.UNIT, n_gpus=1, steps=100, warmup=3,
        ms_per_step=2.2968815970420837, higher_is_better=True, scaling="weak", vs_baseline=None, dtype="f32",
        data="synthetic (seeded Sedov lattice; no dataset)", config=dict(stage, workload="w" * 200),
        pair_interactions_per_s=114383521553.0208, autotune=dict(trial, trials=[trial] * 20), clocks=clocks,
        e2e=dict(value=613876670.1386665, unit=bench.UNIT, h2d_bytes_per_step=117440516,
                 d2h_bytes_per_step=167772164, steps=10, note="n" * 80),
        gpu_launches=4400, roofline=roof, stage_ms_per_step=stage, work_per_step=stage,
        cpu_baseline=dict(value=345.7, unit=bench.UNIT, cores=16, kind="oracle", sample="s" * 150),
        batched=dict(leg, batched_over_plain=3.4), adjoint=dict(leg, forward_value=5e8, forward_backward_value=1e8),
        plummer=dict(leg, ms_per_evaluation=25.9), tube=dict(leg, ms_per_step=2.5),
        block=dict(leg, global_ms=17.6, block_ms=5.4, speedup=3.2))


def test_line_is_short_and_keeps_the_headline():
    rec = _record()
    line = bench.headline(rec)
    assert len(json.dumps(rec)) > 15000 and len(json.dumps(line)) < 2600
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches"):
        assert line[k] == rec[k], k
    assert line["clocks"] == {k: rec["clocks"][k] for k in ("sm_mhz", "sm_max_mhz", "reasons", "samples")}
    assert line["block"]["speedup"] == 3.2 and "autotune" not in line["batched"]
    assert bench.headline(dict(rec, tube=None, plummer={}))["value"] == rec["value"]
