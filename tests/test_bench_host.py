"""Host-side logic of bench.py that needs no GPU: the hash that ties the committed DRAM traffic
to the seeding kernels' code."""
import json

import pytest

import bench


def test_kernel_hash_ignores_comments_and_blank_lines():
    src = '''// a comment
#include "x.h"   /* a block
comment */
int f(int a) {  // trailing
    const char *s = "// not a comment /* nor this */";

    return a + '/';
}
'''
    same = '''#include "x.h"
int f(int a) {
    const char *s = "// not a comment /* nor this */";
    return a + '/';
}'''
    assert bench.strip_comments(src) == same
    assert bench.strip_comments(src.replace("return a + '/'", "return a - '/'")) != same


def full_report():
    """A report of the size that a whole run makes: a 92-point autotuner grid, load sweep, counters."""
    shape = dict(block_size=512, work_queue=True, smem_form="slots", smem_burst=16, smem_wait=8, smem_warps=None,
                 smem_reads_per_warp=64, locate_walks_per_lane=16, locate_join=False, locate_aux=False, ms=11.185)
    x = 447051822.29417205
    return {
        "metric": bench.METRIC, "value": x, "unit": "reads/s", "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": x,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
        "config": {"workload": bench.WORKLOADS[3], **{f"size_{i}": 20_000_000 for i in range(13)},
                   "l2": "inputs larger than L2 (reads 3 GB; index blocks 1 GB, 14-mer table 3.2 GB)"},
        "smems_per_s": x, "hits_per_s": x,
        "roofline": {**{k: x for k in bench.SHORT_KEYS["roofline"]}, "gather_ceiling": {f"g{i}": x for i in range(9)},
                     "kernels": {k: {"ms_per_launch": x, "bytes": 1 << 40, "GBps": x} for k in ("smem", "locate")}},
        "cpu_baseline": {"value": x, "unit": "reads/s", "cores": 16, "kind": "oracle", "sample": "s" * 120,
                         "single_core": {"value": x}, "batched_prefetch": {"value": x, "sample": "s" * 100}},
        "e2e": {"value": x, "unit": "reads/s", "h2d_bytes_per_step": 3160000008, "d2h_bytes_per_step": 2959135480,
                "call": "c" * 110, "note": "n" * 100, "identical_output": True},
        "gpu_launches": 1380,
        "forms": {"plain_launch": {"ms_per_step": x, "reads_per_s": x}, "graph_plan": {"ms_per_step": x, "shape": shape},
                  "reported": "graph_plan", "graph_plan_locate_aux": {"ms_per_step": x, "shape": shape}},
        "batched": {**{k: x for k in bench.SHORT_KEYS["batched"]}, "autotune_grid": [shape] * 92, "autotuned": shape},
        "rescue_prefilter": {"pairs_per_s": x, "kernel_ms": x, "workload": "w" * 150, "roofline": {"ops": "o" * 60}},
        "served": {**{k: x for k in bench.SHORT_KEYS["served"]}, "load_sweep": [{f"v{i}": x for i in range(6)}] * 4,
                   "server_counters": {f"c{i}": 1 << 30 for i in range(13)}},
        "bisulfite": {"reads": 1, "hits": 45083658, "ms": {k: x for k in ("seed", "locate", "filter", "split")},
                      "whole_bs_path_reads_per_s": x, "workload": "w" * 150},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 11},
    }


def test_line_on_stdout_is_short_and_keeps_the_headline():
    """A line of 29 kB was cut by a reader that keeps the end of the output; every headline key stays whole."""
    full = full_report()
    assert len(json.dumps(full)) > 20_000
    line = json.loads(json.dumps(bench.short_line(full)))
    assert len(json.dumps(line)) < bench.SHORT_MAX
    assert set(line) == set(full)
    for k in full:
        if k not in bench.SHORT_KEYS and k != "forms":
            assert line[k] == full[k], k
    for part, keys in bench.SHORT_KEYS.items():
        assert set(keys) <= set(line[part])
    assert line["e2e"]["h2d_bytes_per_step"] == 3160000008
    assert bench.short_line(dict(full, e2e=None, batched=None, cpu_baseline=None))["e2e"] is None


def test_run_shape_leaves_out_what_has_no_effect():
    mb = pytest.importorskip("paper_2606_15357_gb300")
    a = mb.run_shape(mb.Opts(block_size=512, smem_burst=4, smem_wait=16, smem_reads_per_warp=40, prefetch_depth=2))
    b = mb.run_shape(mb.Opts(block_size=512, flags=mb.MB_BATCHED | mb.MB_LOCATE_JOIN))
    assert a == b and a["work_queue"] and a["smem_reads_per_warp"] == 64 and "smem_burst" not in a
    assert mb.shape_of(mb.Opts(smem_reads_per_warp=32))["smem_reads_per_warp"] == 64
    assert mb.shape_of(mb.Opts(smem_reads_per_warp=31))["smem_reads_per_warp"] == 31
    assert not mb.run_shape(mb.Opts(flags=mb.MB_SMEM_ONE_LOOP))["work_queue"]
