"""What bench.py says about the launches of a step."""
import pytest

import bench
import lightkv_synth as S


def test_no_kernel_is_reported_that_the_engine_does_not_launch():
    assert "window_build" not in bench.kernel_names("auto") and len(bench.kernel_names("auto")) == 5
    assert bench.kernel_names("simt")[0] == "window_build" and len(bench.kernel_names("simt")) == 6


@pytest.mark.gpu
@pytest.mark.parametrize("engine,in_place", [("auto", False), ("auto", True), ("simt", False)])
def test_launches_are_the_kernels_a_step_really_launches(engine, in_place):
    import torch
    import __graft_entry__ as entry
    entry.build()
    import paper_2605_00789_b200 as L
    wl = S.workload("small")
    plan = L.Plan(wl.batch, wl.hidden, wl.n_q_heads, wl.n_kv_heads, wl.head_dim, wl.n_layers, wl.tiles, wl.layers,
                  wl.windows, wl.keep, wl.n_text, engine=L.ENGINE_AUTO if engine == "auto" else L.ENGINE_SIMT)
    stages = bench.build_inputs(wl, plan, L, torch, torch.device("cuda"), sample_offset=0)
    for s in stages:
        s["kv_in_place"] = in_place
    step = lambda: bench.run_step(L, plan, wl, stages)
    step()
    assert bench.count_launches(step) == len(stages) * len(bench.kernel_names(engine))
