"""The printed line's sub-results are short: what collects the line may keep only its last
kilobytes."""
import json

import bench

ROOF = {"bound": "hbm", "achieved": 5493.478015783379, "peak": 6800.0, "unit": "GB/s", "frac": 0.8078644140857911,
        "traffic": None, "kernel": "d2q9 batched step kernel (2048 lattices, 80765115 nodes, fp32)", "note": "x" * 400}
WORK = {"mlups": 92558.89388204365, "ms_per_step": 1.7451616287231446, "steps": 20, "nodes": 161530230,
        "gpu_launches": 40, "roofline": ROOF, "all_kernels": [ROOF, ROOF], "l2": "state larger than L2", "workload": "w" * 60}
FP64 = dict(WORK, roofline=dict(ROOF, bound="alu", frac=4.63973528154141, hbm={"frac": 0.6422700660888235}))
LREF = {"mlups": 1.0 / 3, "ms_per_step": 2.0 / 3, "steps": 40, "step_kernel": {"ms": 0.3, "roofline": ROOF}}
TTS = {"steps": 10200, "seconds": 0.017846688000020094, "l2_vs_fp64_steady": 9.643857734457967e-05, "reached": True,
       "criterion": "c" * 150, "launch": "l" * 80}
SWEEP = {"seconds": 0.41320195200000853, "steps": [400, 1600, 6400, 25600, 102400],
         "l2_vs_closed_form": [0.008194371557341021] * 5, "orders": [-0.3751013603442858] * 4}


def _ext():
    return {"storages": {"grid": "512^3", "run_steps": 1000, "fp64": {"run": {"mlups": 1.0 / 3}, "u_max": 1.0 / 3},
                         **{s: dict(WORK, run={"mlups": 1.0 / 3}, l2_u_vs_fp64=1.0 / 7) for s in ("fp32", "fp16", "bf16")}},
            "workloads": {**{f"workload_number_{k}": FP64 if k % 3 == 0 else WORK for k in range(13)}, "lref": LREF,
                          "broken": {"error": "e"}},
            "time_to_solution": {**{f"poiseuille_case_{k}": TTS for k in range(11)},
                                 **{f"cde_sweep_case_{k}": SWEEP for k in range(10)},
                                 "batched_sweep_subset": {"members": {"d2q9_channels": 32}, "criterion": "c" * 200,
                                                          "fp64_batched": TTS, "fp32_batched_graph": TTS}},
            "extras_seconds": 39.56719593600002}


def test_sub_results_are_short_and_hold_the_figures():
    b = bench.brief(_ext())
    assert len(json.dumps(b)) <= 6000 < len(json.dumps(_ext()))
    assert b["workloads"]["workload_number_0"]["frac"] == {"alu": 4.6397, "hbm": 0.64227}
    assert b["workloads"]["workload_number_1"]["mlups"] == 92559.0 and b["workloads"]["broken"] == {"error": "e"}
    assert b["workloads"]["lref"]["frac"] == {"hbm": 0.80786}
    assert b["storages"]["fp16"]["l2_u_vs_fp64"] == 0.14286 and b["storages"]["grid"] == "512^3"
    assert b["time_to_solution"]["poiseuille_case_3"] == {"seconds": 0.017847, "steps": 10200, "reached": True,
                                                          "l2_vs_fp64_steady": 9.6439e-05}
    assert b["time_to_solution"]["cde_sweep_case_2"]["orders"] == [-0.3751] * 4
    assert b["time_to_solution"]["batched_sweep_subset"]["fp64_batched"]["reached"] is True
