"""bench.py names the kernels, launches and bytes that the library's plans
say, not those of its default workload."""
import types

import bench
from paper_1107_4543_gb300 import lbm


def test_kernel_names_follow_the_plan():
    k = bench.step_kernel
    assert k(lbm, "f32", lbm.LBM_PLAN_ROWS, batched=True) == "k_rows_batch<float>"
    assert k(lbm, "f16", lbm.LBM_PLAN_SINGLE, batched=True) == "k_step_batch<__half>"
    assert k(lbm, "bf16", lbm.LBM_PLAN_SINGLE) == "k_step_dev<__nv_bfloat16>"
    assert k(lbm, "f32", lbm.LBM_PLAN_TILES) == "k_step_tile<float>"
    assert k(lbm, "f64dev", lbm.LBM_PLAN_SINGLE) == "k_step_dev<double>"
    assert k(lbm, "f64", lbm.LBM_PLAN_SINGLE) == "k_step_f64"


def test_bytes_follow_the_steps_per_launch():
    assert bench.hbm_bytes_per_update("f32", 1) == 72
    assert bench.hbm_bytes_per_update("f16", 3) == 12


def test_resident_launches_count_the_kinds():
    def specs(*nodes):
        return [{"nx": n, "ny": 1} for n in nodes]

    n = bench.resident_launches
    assert n(specs(100, 5000), [False, False], "f32") == 0
    assert n(specs(1024, 3000), [True, True], "f32") == 1
    assert n(specs(100, 1024, 3220, 9000), [True, True, True, False], "f32") == 3
    assert n(specs(100, 1024, 6440), [True, True, True], "f16") == 2


def test_operation_fraction():
    props = types.SimpleNamespace(multi_processor_count=100)
    torch = types.SimpleNamespace(cuda=types.SimpleNamespace(get_device_properties=lambda d: props))
    # 97 operations per update, 100 SMs of 128 per clock at 1 GHz
    r = bench.alu_record(torch, "f32", 12.8e12 / 97 / 1e6, 1000.0)
    assert r["frac"] == 1.0 and r["ops_per_update"] == 97
