"""The roofline arithmetic of bench.py against numbers worked out by hand (no GPU, no weights generated)."""
import types

import bench
from paper_2511_11346_b200 import inputs as I


def _fake(shape, T):
    return types.SimpleNamespace(shape=shape, T=T, name="fake", wpp=0)


def test_algorithmic_flops_of_the_mixture_training_head():
    # 2 d (n r v + S r) per position: 2 * 4096 * (8*16*320 + 1*16) = 335 675 392 FLOP, times 8192 positions
    wl = _fake(I.HeadShape(I.CP, 8, 16, 320, 4096), 8192)
    assert bench.algorithmic_flops(wl) == 2 * 4096 * (40960 + 16) * 8192 == 2749852811264


def test_algorithmic_flops_count_every_sum_unit_of_the_tree():
    # S = 1 + (n - 2) r = 449 sum units of r = 32 inputs
    wl = _fake(I.HeadShape(I.BTREE, 16, 32, 320, 4096), 4096)
    assert bench.algorithmic_flops(wl) == 2 * 4096 * (16 * 32 * 320 + 449 * 32) * 4096


def test_circuit_bytes():
    # the circuit kernel reads G [T, n, r] and log omega [T, S r] and writes [T], fp32
    wl = _fake(I.HeadShape(I.CP, 8, 16, 320, 4096), 8192)
    assert bench.circuit_bytes(wl) == 4 * 8192 * (128 + 16 + 1) == 4751360
    wl = _fake(I.HeadShape(I.HMM_CTX, 16, 32, 320, 4096), 8192)
    assert bench.circuit_bytes(wl) == 4 * 8192 * (512 + (1 + 15 * 32) * 32 + 1)


def test_workload_name_states_the_shape():
    wl = _fake(I.HeadShape(I.CP, 8, 16, 320, 4096), 8192)
    name = bench.workload_name(1, wl)
    for piece in ("T=8192", "d=4096", "n=8", "r=16", "v=320"):
        assert piece in name


def test_cpu_baseline_helper_runs_the_oracle_on_a_sample():
    wl = I.config_workload(0)
    rate, seconds = bench.oracle_positions_per_s(wl, 32, chunk=16)
    assert rate > 0 and seconds > 0 and abs(rate * seconds - 32) < 1e-6
    assert bench.host_threads() >= 1


def test_the_printed_line_keeps_the_headline_and_stays_short():
    import json
    cell = {"workload": "decode_cp_n8_P1: P=1 wpp=16 d=4096 n=8 r=16 v=320", "windows_per_s": 234686.7015776039, "p50_ms": 0.06817599758505821,
            "calls": 200, "kernels_per_call": 3, "kernel_p50_ms": [0.05974400043487549] * 3, "device_status": 0,
            "cuda_graph_replay": {"p50_ms": 0.06543999910354614, "hbm_frac": 0.77135548972915, "note": "n" * 80},
            "draft_plus_accept": {"p50_ms": 0.07708799839019775, "calls": "c" * 60},
            "hbm_roofline": {"frac": 0.7403999111771542, "weight_pass_kernel_frac": 0.8448965952893371, "note": "n" * 60}}
    other = {"workload": "hmm_train: T=8192", "positions_per_s": 2322842.4582707235, "positions_per_s_sustained": 2048571.31,
             "roofline": {"frac": 0.9900891797413823, "peak_source": "p" * 120}, "draft_whole_batch": {"ms_per_call": 2.6565343856811525}}
    line = {"metric": bench.METRIC, "value": 4689615.306671511, "unit": bench.UNIT, "ms_per_step": 1.74683837890625,
            "e2e": {"value": 4045460.1672665244}, "roofline": {"frac": 0.99967167093412, "sustained": {"frac": 0.99912475901711}},
            "workloads": [other, dict(other)], "decode_sweep": [dict(cell) for _ in range(12)], "draft": cell, "draft_whole_batch": None,
            "backward": {"ms_per_call": 6.7123456789, "phases": "p" * 300}}
    out = bench.printed_line(line)
    text = json.dumps(out)
    assert "\n" not in text and len(text) < 3000
    for key in ("metric", "value", "unit", "ms_per_step", "e2e"):
        assert out[key] == line[key]
    assert len(out["decode"]) == 12 and out["decode"][0] == ["decode_cp_n8_P1", 0.068176, 0.06544, 0.077088, 0.7404, 0.844897]
    assert len(out["decode_columns"]) == len(out["decode"][0])
    assert [w["draft_whole_batch_ms"] for w in out["workloads"]] == [2.65653] * 2 and out["backward_ms"] == 6.71235
    assert "decode_sweep" not in out and "draft" not in out and len(line["decode_sweep"]) == 12
