"""Parity of the CUDA path (through the C ABI) with the CPU oracle on seeded synthetic inputs.

Index sets (survivors, dst, positions, counts, group lists) must be bit-exact on inputs whose
selection margins are >= 1e-3; merged hidden states and K/V within max-abs 2e-2 and relative 1e-2
(bf16 storage, fp32 accumulation) or 1e-5 relative (fp32 mode)."""
import dataclasses

import numpy as np
import pytest

import lightkv_synth as S
from tests import harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    import __graft_entry__ as entry
    assert torch.cuda.is_available()
    entry.build()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("engine", ["simt", "auto"])
@pytest.mark.parametrize("xi_mode", ["attn", "lse", "given", "uniform"])
def test_tiny_schedule(dtype, engine, xi_mode):
    stats = H.run_schedule(S.workload("tiny"), dtype=dtype, xi_mode=xi_mode, engine=engine)
    assert [s["n_out"] for s in stats] == [[20, 20], [15, 15], [8, 8]]


@pytest.mark.parametrize("dtype,engine", [("bf16", "simt"), ("bf16", "auto"), ("fp32", "simt")])
def test_small_ragged_multitile_gqa(dtype, engine):
    # two tiles of different shape, windows that do not divide the grid, GQA, keep 0.55 / 0.6 / 0.5
    H.run_schedule(S.workload("small"), dtype=dtype, engine=engine)


@pytest.mark.parametrize("kv_mode,paged", [("gather", 0), ("merge", 16), ("gather", 16), ("merge", 5)])
def test_small_kv_modes_and_paged_cache(kv_mode, paged):
    H.run_schedule(S.workload("small"), kv_mode=kv_mode, paged=paged, stages=[0])


def test_small_lse_mode_on_tensor_cores():
    # row log-sum-exp supplied by the caller: only the prompt key tiles are visited (tcgen05 path, GQA)
    H.run_schedule(S.workload("small"), xi_mode="lse")
    wl = dataclasses.replace(S.workload("cfg0"), n_text=200)      # prompt keys spanning two key tiles
    H.run_schedule(wl, xi_mode="lse")


@pytest.mark.parametrize("kv_mode", ["merge", "gather"])
def test_small_token_major_kv_cache(kv_mode):
    # K/V stored [B, N, H_kv, dh]: the same call with other strides
    H.run_schedule(S.workload("small"), kv_mode=kv_mode, kv_layout="bnhd", stages=[0, 1])


@pytest.mark.parametrize("w", [4, 6, 1])
@pytest.mark.parametrize("engine", ["simt", "auto"])
def test_cfg0_single_step(w, engine):
    wl = dataclasses.replace(S.workload("cfg0"), windows=(w,))
    stats = H.run_schedule(wl, engine=engine)
    assert stats[0]["n_out"] == [{4: 320, 6: 324, 1: 317}[w]]


@pytest.mark.parametrize("name", ["cfg1", "cfg1r"])
def test_cfg1_full_schedule(name):
    stats = H.run_schedule(S.workload(name))
    if name == "cfg1":
        assert [s["n_out"] for s in stats] == [[288], [144], [72]]


@pytest.mark.parametrize("name", ["small", "cfg1"])
def test_second_stream_inside_compress_layer(name):
    # window build + FD on aux_stream beside xi: same results as the oracle, run after run
    import torch
    aux = torch.cuda.Stream()
    for _ in range(2):
        H.run_schedule(S.workload(name), aux_stream=aux)


@pytest.mark.parametrize("name", ["small", "cfg1"])
def test_kv_compaction_behind_the_map_event(name):
    # lightkv_compact_kv on a second stream behind map_event (recorded once the merge map is complete, before
    # the hidden-state merge), together with the second stream inside the call
    import torch
    aux, kv_stream = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(2):
        H.run_schedule(S.workload(name), aux_stream=aux, kv_stream=kv_stream)


def test_cfg0_fp32_mode():
    H.run_schedule(dataclasses.replace(S.workload("cfg0"), hidden=1024, n_q_heads=8, n_kv_heads=8), dtype="fp32")


def test_text_after_and_prompt_subrange():
    wl = S.workload("small")
    plan = H.make_plan(wl)
    inp = H.prepare_stage(wl, 0)
    # move the last 4 text rows behind the vision block: [15 text | vision | 4 text], J = [2, 12)
    vb, after = wl.n_text - 4, 4
    for key in ("hidden", "q", "k", "v"):
        a = inp[key]
        axis = 1 if key == "hidden" else 2
        a = np.concatenate([np.take(a, range(0, vb), axis), np.take(a, range(wl.n_text, a.shape[axis]), axis),
                            np.take(a, range(vb, wl.n_text), axis)], axis)
        inp[key] = np.ascontiguousarray(a)
    inp["vis_begin"] = vb
    assert len(set(inp["n_vis"])) == 1        # full grids: every sample has the same length here
    gpu = H.gpu_stage(plan, wl, 0, inp, n_text_after=after, text_range=(2, 12))
    ref = H.oracle_stage(wl, 0, inp, n_text_after=after, text_range=(2, 12))
    H.compare_stage(wl, 0, inp, ref, gpu, n_text_after=after)
    for b, r in enumerate(ref):
        n_out = int(r["n_out"])
        np.testing.assert_array_equal(gpu["hidden_out"][b, vb + n_out:vb + n_out + after],
                                      inp["hidden"][b, vb + int(inp["n_vis"][b]):][:after])


def test_ragged_batch_and_empty_sample():
    wl = S.workload("small")
    plan = H.make_plan(wl)
    full = np.arange(wl.n_vis, dtype=np.int32)
    rng = np.random.default_rng(5)
    pos = [full, np.sort(rng.choice(full, 97, replace=False)).astype(np.int32), full[:0]]
    inp = H.prepare_stage(wl, 0, pos)
    gpu = H.gpu_stage(plan, wl, 0, inp)
    ref = H.oracle_stage(wl, 0, inp)
    H.compare_stage(wl, 0, inp, ref, gpu)
    assert int(gpu["n_vis_out"][2]) == 0


def test_keep_one_is_identity_on_device():
    wl = dataclasses.replace(S.workload("small"), keep=(1.0, 1.0, 1.0))
    plan = H.make_plan(wl)
    inp = H.prepare_stage(wl, 0, repair=False)
    gpu = H.gpu_stage(plan, wl, 0, inp)
    n = wl.n_vis
    assert (gpu["n_vis_out"] == n).all()
    np.testing.assert_array_equal(gpu["hidden_out"][:, :wl.n_text + n], inp["hidden"])
    np.testing.assert_array_equal(gpu["k_out"][:, :, :wl.n_text + n], inp["k"])
    np.testing.assert_array_equal(gpu["dst"][:, :n], np.tile(np.arange(n), (wl.batch, 1)))
    assert (gpu["weight"][:, :n] == 1.0).all()


def test_device_status_word_flags_unsorted_positions():
    wl = S.workload("tiny")
    plan = H.make_plan(wl, xi_mode="uniform")
    inp = H.prepare_stage(wl, 0, repair=False)
    inp["pos"][1, [3, 4]] = inp["pos"][1, [4, 3]]
    gpu = H.gpu_stage(plan, wl, 0, inp, xi_mode="uniform")
    assert int(gpu["status"][0]) & 1


def test_vanishing_xi_gives_the_group_mean_and_the_status_bit():
    # xi = 0 for every token of sample 0: the sum over a group vanishes, the merge falls back to the plain
    # group mean (as the oracle does) and the ZERO_WEIGHT bit is raised; the other samples are unaffected
    wl = S.workload("small")
    plan = H.make_plan(wl, xi_mode="given")
    inp = H.prepare_stage(wl, 0)
    inp["xi"] = np.random.default_rng(5).uniform(0.05, 3.0, size=inp["pos"].shape).astype(np.float32)
    inp["xi"][0] = 0.0
    gpu = H.gpu_stage(plan, wl, 0, inp, xi_mode="given")
    ref = H.oracle_stage(wl, 0, inp, "given")
    H.compare_stage(wl, 0, inp, ref, gpu, expect_status=2)
    plan.close()


def test_run_to_run_bit_repeatability():
    wl = S.workload("small")
    plan = H.make_plan(wl)
    inp = H.prepare_stage(wl, 0, repair=False)
    a = H.gpu_stage(plan, wl, 0, inp)
    b = H.gpu_stage(plan, wl, 0, inp)
    for key in ("hidden_out", "k_out", "v_out", "weight", "xi_out", "dst", "grp_src", "grp_off", "pos_out"):
        np.testing.assert_array_equal(a[key], b[key])


# ---- prompt ranges, rows without the causal mask, the row log-sum-exp as an output ---------------------------

@pytest.mark.parametrize("engine", ["simt", "auto"])
def test_prompt_ranges_bidirectional_rows_and_lse_out(engine):
    wl = S.workload("small")                                   # 19 text rows, head_dim 128 (tcgen05 with "auto")
    H.run_schedule(wl, engine=engine, stages=[0], text_ranges=[(1, 4), (7, 8), (10, 19)], want_lse=True)
    H.run_schedule(wl, engine=engine, stages=[0, 1], bidirectional=True, want_lse=True)
    H.run_schedule(wl, engine=engine, stages=[0], bidirectional=True, xi_mode="lse", text_ranges=[(0, 3), (9, 19)])


def test_prompt_ranges_over_several_key_tiles():
    # 200 prompt rows = four 64-key tiles; J = three ranges with holes, cut by tile borders
    wl = dataclasses.replace(S.workload("cfg0"), n_text=200, hidden=256)
    ranges = [(3, 50), (60, 70), (100, 190)]
    H.run_schedule(wl, text_ranges=ranges, want_lse=True)
    H.run_schedule(wl, text_ranges=ranges, xi_mode="lse")
    H.run_schedule(wl, text_ranges=ranges, bidirectional=True, want_lse=True)


def test_bidirectional_rows_with_text_behind_the_vision_block():
    # [15 text | vision | 4 text], no causal mask: the rows behind the vision block are keys too (not in J)
    wl = S.workload("small")
    plan = H.make_plan(wl)
    inp = H.prepare_stage(wl, 0)
    vb, after = wl.n_text - 4, 4
    for key in ("hidden", "q", "k", "v"):
        a = inp[key]
        axis = 1 if key == "hidden" else 2
        a = np.concatenate([np.take(a, range(0, vb), axis), np.take(a, range(wl.n_text, a.shape[axis]), axis),
                            np.take(a, range(vb, wl.n_text), axis)], axis)
        inp[key] = np.ascontiguousarray(a)
    inp["vis_begin"] = vb
    gpu = H.gpu_stage(plan, wl, 0, inp, n_text_after=after, text_range=(2, 12), bidirectional=True, want_lse=True)
    ref = H.oracle_stage(wl, 0, inp, n_text_after=after, text_range=(2, 12), causal=False)
    H.compare_stage(wl, 0, inp, ref, gpu, n_text_after=after)
    H.check_lse_out(inp, gpu, wl.n_q_heads, wl.n_kv_heads, range(wl.batch), causal=False, n_text_after=after)


@pytest.mark.parametrize("name", ["small", "cfg1"])
def test_the_librarys_own_row_lse_feeds_the_lse_mode(name):
    """ATTN_FULL hands out the row log-sum-exp it saw (lse_out); given back as the input of ATTN_LSE, only the
    prompt keys are visited and xi, the merge map and the merged rows agree with ATTN_FULL and the oracle."""
    wl = S.workload(name)
    full, lse_plan = H.make_plan(wl), H.make_plan(wl, xi_mode="lse")
    inp = H.prepare_stage(wl, 0)
    a = H.gpu_stage(full, wl, 0, inp, want_lse=True)
    b = H.gpu_stage(lse_plan, wl, 0, inp, xi_mode="lse", lse=a["lse_out_dev"])
    ref = H.oracle_stage(wl, 0, inp)
    H.compare_stage(wl, 0, inp, ref, a)
    H.compare_stage(wl, 0, inp, ref, b)
    H.check_lse_out(inp, a, wl.n_q_heads, wl.n_kv_heads, range(wl.batch))
    for key in ("dst", "grp_src", "grp_off", "pos_out"):
        np.testing.assert_array_equal(a[key], b[key])
    nv = int(inp["n_vis"][0])
    np.testing.assert_allclose(a["xi_out"][:, :nv], b["xi_out"][:, :nv], rtol=2e-3)


@pytest.mark.parametrize("name", ["small", "cfg1"])
def test_logits_far_above_the_first_tiles_maximum_take_the_safe_pass(name):
    """The tensor-core xi kernel subtracts the maximum of a row's FIRST key tile and checks its sums at the end.
    Here one late key of one KV head is scaled by 128, so that many rows meet a logit far more than 88 above
    that reference: their sums leave the fp32 range, the CTA repeats the item with a running maximum, and the
    result still matches the oracle (the other heads keep xi away from zero)."""
    wl = S.workload(name)
    plan = H.make_plan(wl)
    inp = H.prepare_stage(wl, 0)
    late = inp["vis_begin"] + int(inp["n_vis"].min()) * 2 // 3
    inp["k"][:, 0, late] *= 128.0                              # a power of two: still bf16 values
    logit = inp["q"][0, 0, late + 1:] @ inp["k"][0, 0, late] / np.sqrt(wl.head_dim)
    first = (inp["q"][0, 0, late + 1:] @ inp["k"][0, 0, :64].T / np.sqrt(wl.head_dim)).max(axis=1)
    assert (logit - first > 100).any()                         # the case really leaves the fp32 range
    gpu = H.gpu_stage(plan, wl, 0, inp, want_lse=True)
    del gpu["k_out"], gpu["v_out"]      # the scaled key row is outside the value range the bf16 K/V tolerance is meant for
    H.compare_stage(wl, 0, inp, H.oracle_stage(wl, 0, inp), gpu)
    H.check_lse_out(inp, gpu, wl.n_q_heads, wl.n_kv_heads, range(inp["hidden"].shape[0]), atol=2e-2)
    plan.close()


# ---- K/V compaction inside the cache's own rows / pages ---------------------------------------------------------

@pytest.mark.parametrize("kv_mode,paged,layout", [("merge", 0, "bhnd"), ("gather", 0, "bhnd"), ("merge", 16, "bhnd"),
                                                  ("merge", 5, "bhnd"), ("gather", 16, "bhnd"), ("merge", 0, "bnhd")])
def test_in_place_kv_compaction(kv_mode, paged, layout):
    # destination = source: groups are merged over their surviving token's row, then rows move forward plane by
    # plane; compared with the oracle like the out-of-place form (ragged windows, two tiles, GQA, three stages)
    H.run_schedule(S.workload("small"), kv_mode=kv_mode, paged=paged, kv_layout=layout, kv_in_place=True)


def test_in_place_kv_compaction_long_rows_and_text_behind():
    # 2304 tokens per sample: a plane is swept in many chunks (sources of a chunk lie inside the next chunks'
    # destinations); text rows behind the vision block move forward with it
    wl = S.Workload(name="inpl", config_id=140, batch=2, tiles=((48, 48),), n_text=37, hidden=64, n_q_heads=4,
                    n_kv_heads=2, head_dim=64, n_layers=16, layers=(3, 7), windows=(6, 3), keep=(0.55, 0.5))
    H.run_schedule(wl, xi_mode="given", kv_in_place=True)
    plan = H.make_plan(wl, xi_mode="uniform")
    inp = H.prepare_stage(wl, 0)
    vb, after = wl.n_text - 9, 9
    for key in ("hidden", "q", "k", "v"):
        a = inp[key]
        axis = 1 if key == "hidden" else 2
        a = np.concatenate([np.take(a, range(0, vb), axis), np.take(a, range(wl.n_text, a.shape[axis]), axis),
                            np.take(a, range(vb, wl.n_text), axis)], axis)
        inp[key] = np.ascontiguousarray(a)
    inp["vis_begin"] = vb
    gpu = H.gpu_stage(plan, wl, 0, inp, xi_mode="uniform", n_text_after=after, kv_in_place=True)
    ref = H.oracle_stage(wl, 0, inp, "uniform", n_text_after=after)
    H.compare_stage(wl, 0, inp, ref, gpu, n_text_after=after)
    plan.close()


@pytest.mark.parametrize("batch,n_kv,head_dim,grid,text", [
    (1, 1, 64, (24, 24), 3),         # one plane pair, cut into parts of 64 bytes
    (3, 2, 24, (12, 14), 0),         # rows of three 16-byte pieces: not cut
    (2, 3, 96, (40, 41), 17),        # parts of 64 bytes (rows of twelve pieces)
    (1, 2, 128, (72, 74), 5),        # fits on chip in parts of 32 bytes only
    (1, 2, 128, (80, 82), 5),        # gathered, the survivors' rows fit on chip; to be merged, all rows do not
    (1, 1, 128, (100, 96), 5),       # does not fit: merged at the survivors, then moved in chunks
])
@pytest.mark.parametrize("kv_mode,paged", [("merge", 0), ("gather", 16)])
def test_in_place_planes_over_cuts(batch, n_kv, head_dim, grid, text, kv_mode, paged):
    wl = S.Workload(name="plane", config_id=141, batch=batch, tiles=(grid,), n_text=text, hidden=64, n_q_heads=n_kv,
                    n_kv_heads=n_kv, head_dim=head_dim, n_layers=16, layers=(3,), windows=(3,), keep=(0.55,))
    H.run_schedule(wl, xi_mode="given", kv_mode=kv_mode, paged=paged, kv_in_place=True)


def test_in_place_rows_behind_the_new_end():
    # a merged group replaces its survivor's row also where that row lies behind the new end of the sample; all other
    # rows there keep what they held (the one-kernel form leaves the cache as the merge-then-move form does)
    import torch
    import paper_2605_00789_b200 as L
    wl = dataclasses.replace(S.workload("cfg1"), hidden=64, n_q_heads=2, n_kv_heads=2)
    plan = H.make_plan(wl, xi_mode="uniform")
    inp = H.prepare_stage(wl, 0)
    gpu = H.gpu_stage(plan, wl, 0, inp, xi_mode="uniform")
    k = H.to_device(inp["k"], "bf16")
    v = H.to_device(inp["v"], "bf16")
    L.compact_kv(plan, 0, gpu["out"], k, v, k, v, vis_begin=wl.n_text)
    got = k.float().cpu().numpy()[0]
    n_out, off, src = int(gpu["n_vis_out"][0]), gpu["grp_off"][0], gpu["grp_src"][0]
    want = inp["k"][0].copy()
    for o in range(n_out):
        if off[o + 1] - off[o] > 1:
            want[:, wl.n_text + src[off[o]]] = gpu["k_out"][0][:, wl.n_text + o]
    np.testing.assert_array_equal(got[:, wl.n_text + n_out:], want[:, wl.n_text + n_out:])
    plan.close()


def test_in_place_equals_out_of_place_bit_for_bit():
    wl = S.workload("cfg1")
    plan = H.make_plan(wl)
    inp = H.prepare_stage(wl, 0, repair=False)
    a = H.gpu_stage(plan, wl, 0, inp)
    b = H.gpu_stage(plan, wl, 0, inp, kv_in_place=True)
    np.testing.assert_array_equal(a["k_out"], b["k_out"])
    np.testing.assert_array_equal(a["v_out"], b["v_out"])
    plan.close()


# ---- packed (ragged) batches: samples back to back on one row axis ----------------------------------------------

@pytest.mark.parametrize("engine,xi_mode,in_place", [("auto", "attn", False), ("simt", "attn", False),
                                                     ("auto", "lse", False), ("auto", "attn", True)])
def test_packed_batch_with_row_offsets(engine, xi_mode, in_place):
    """Three samples of different lengths (one of them empty) stored without padding: every tensor has one row
    axis and seq_start / seq_start_out say where a sample begins.  Same results as the padded form."""
    import torch
    import paper_2605_00789_b200 as L
    wl = S.workload("small")
    plan = H.make_plan(wl, xi_mode=xi_mode, engine=engine)
    full = np.arange(wl.n_vis, dtype=np.int32)
    rng = np.random.default_rng(6)
    pos = [full, np.sort(rng.choice(full, 101, replace=False)).astype(np.int32), full[:0]]
    inp = H.prepare_stage(wl, 0, pos)
    info = plan.stage_info(0)
    vb, bsz = inp["vis_begin"], 3
    lens = [vb + int(n) for n in inp["n_vis"]]
    start = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    start_out = (np.arange(bsz + 1) * (vb + info.cap_out)).astype(np.int32)
    dev = "cuda"

    def pack(a, axis):          # [B, (H,) N, w] -> [1, (H,) total, w]
        return np.concatenate([np.take(a[b], range(lens[b]), axis - 1) for b in range(bsz)], axis - 1)[None]

    hid = H.to_device(pack(inp["hidden"], 1), "bf16", dev)
    q, k, v = (H.to_device(pack(inp[n], 2), "bf16", dev) for n in ("q", "k", "v"))
    out = L.StageBuffers(plan, 0, vb + info.cap_out, dev)
    hidden_out = torch.full((1, int(start_out[-1]), wl.hidden), float("nan"), dtype=torch.bfloat16, device=dev)
    pos_pad = np.pad(inp["pos"], ((0, 0), (0, info.cap_in - inp["pos"].shape[1])), constant_values=-1)
    kw = dict(vis_begin=vb, q=q, k=k, n_vis=torch.from_numpy(inp["n_vis"]).to(dev), pos=torch.from_numpy(pos_pad).to(dev),
              seq_start=torch.from_numpy(start[:-1].copy()).to(dev), seq_start_out=torch.from_numpy(start_out[:-1].copy()).to(dev),
              hidden_out=hidden_out)
    if xi_mode == "lse":
        lse = H.oracle_lse(inp, wl.n_q_heads, wl.n_kv_heads)                      # [B, H, N] padded
        kw["lse"] = torch.from_numpy(pack(lse[:, :, :, None], 2)[..., 0].astype(np.float32)).to(dev)   # [1, H, total]
    L.compress_layer(plan, 0, hid, out, **kw)
    if in_place:
        k_dst, v_dst, dst_start = k, v, kw["seq_start"]
    else:
        k_dst = torch.full((1, wl.n_kv_heads, int(start_out[-1]), wl.head_dim), float("nan"), dtype=torch.bfloat16, device=dev)
        v_dst, dst_start = k_dst.clone(), kw["seq_start_out"]
    L.compact_kv(plan, 0, out, k, v, k_dst, v_dst, vis_begin=vb, n_vis=kw["n_vis"], src_seq_start=kw["seq_start"],
                 dst_seq_start=dst_start)
    torch.cuda.synchronize()
    gpu = {name: getattr(out, name).cpu().numpy() for name in
           ("n_vis_out", "pos_out", "dst", "weight", "grp_off", "grp_src", "xi_out", "status")}
    n_out = gpu["n_vis_out"]
    ho = hidden_out.float().cpu().numpy()[0]
    kd, vd = k_dst.float().cpu().numpy()[0], v_dst.float().cpu().numpy()[0]
    so = start if in_place else start_out
    gpu["hidden_out"] = np.stack([ho[start_out[b]:start_out[b] + vb + info.cap_out] for b in range(bsz)])
    rows = vb + info.cap_out
    gpu["k_out"] = np.stack([np.pad(kd[:, so[b]:so[b] + vb + n_out[b]], ((0, 0), (0, rows - vb - n_out[b]), (0, 0))) for b in range(bsz)])
    gpu["v_out"] = np.stack([np.pad(vd[:, so[b]:so[b] + vb + n_out[b]], ((0, 0), (0, rows - vb - n_out[b]), (0, 0))) for b in range(bsz)])
    ref = H.oracle_stage(wl, 0, inp, xi_mode)
    H.compare_stage(wl, 0, inp, ref, gpu)
    plan.close()


# ---- the variants the paper ablates: Euclidean pair scores, reverse message direction ---------------------------

@pytest.mark.parametrize("metric", ["l2sq", "l2"])
@pytest.mark.parametrize("dtype,engine", [("bf16", "auto"), ("bf16", "simt"), ("fp32", "simt")])
def test_euclidean_pair_scores(metric, dtype, engine):
    H.run_schedule(S.workload("small"), dtype=dtype, engine=engine, metric=metric)
    if dtype == "bf16" and metric == "l2sq":
        H.run_schedule(S.workload("cfg1"), engine=engine, metric=metric)      # windows of 36 / 72 / 144 tokens


@pytest.mark.parametrize("engine", ["simt", "auto"])
def test_reverse_direction_b_into_a(engine):
    # odd windows: the destinations (A) outnumber the sources (B); keep 0.5 on even windows removes all of B
    H.run_schedule(S.workload("small"), engine=engine, direction="b2a")
    H.run_schedule(S.workload("tiny"), engine=engine, direction="b2a", xi_mode="given")
    stats = H.run_schedule(S.workload("cfg1"), engine=engine, direction="b2a")
    assert [s["n_out"] for s in stats] == [[288], [144], [72]]
    H.run_schedule(S.workload("cfg1r"), engine=engine, direction="b2a", metric="l2sq", stages=[0, 1])


# ---- persistent CTAs that take more than one work item ---------------------------------------------------------

def _sm_count():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("head_dim", [64, 128])
def test_lse_mode_persistent_ctas_walk_several_items(head_dim):
    # 4 samples x 8 heads x 16 query tiles = 512 work items for 2 CTAs per SM: most CTAs of the xi kernel
    # take a second item (its barriers and rings run on across items); 130 prompt rows span three key tiles
    wl = S.Workload(name="lsewalk", config_id=130, batch=4, tiles=((64, 32),), n_text=130, hidden=64, n_q_heads=8,
                    n_kv_heads=4, head_dim=head_dim, n_layers=16, layers=(3,), windows=(4,), keep=(0.5,))
    assert 16 * wl.n_q_heads * wl.batch > 3 * _sm_count()
    H.run_schedule(wl, xi_mode="lse")
    H.run_schedule(wl, xi_mode="lse", text_ranges=[(2, 60), (70, 129)])


@pytest.mark.parametrize("head_dim,grid,text,batch,heads", [
    (8, (1, 2), 1, 1, 1),           # less than a query tile; two of four warps have no dimension of the head
    (72, (4, 8), 32, 2, 2),         # one full query tile; keys end on a tile; slices end within the head's last piece
    (80, (3, 11), 63, 2, 4),        # a query more than a tile
    (256, (8, 9), 57, 3, 2),        # largest head: one CTA per SM
    (64, (24, 24), 35, 4, 4),       # 288 CTAs: two per SM, paired from both ends
    (128, (24, 25), 5, 4, 4),       # 304 CTAs: more than are resident
])
@pytest.mark.parametrize("xi_mode", ["attn", "lse"])
def test_xi_fma_tiles(head_dim, grid, text, batch, heads, xi_mode):
    wl = S.Workload(name="xifma", config_id=142, batch=batch, tiles=(grid,), n_text=text, hidden=64, n_q_heads=heads,
                    n_kv_heads=heads if heads < 4 else 2, head_dim=head_dim, n_layers=16, layers=(3,), windows=(1,),
                    keep=(0.55,))
    H.run_schedule(wl, xi_mode=xi_mode, dtype="fp32", engine="simt")
    H.run_schedule(wl, xi_mode=xi_mode, dtype="bf16", engine="simt")


@pytest.mark.parametrize("head_dim,text_ranges", [(64, None), (128, [(32, 96)]), (128, [(0, 64), (96, 129)])])
def test_xi_items_taken_over_and_repeated(head_dim, text_ranges):
    # 4 samples x 8 heads x 16 query tiles = 512 items for the 2 CTAs per SM that are resident: CTAs take over the
    # items of others; one late key of a KV head is scaled so that a quarter of the items leave the fp32 range and are
    # repeated from the CTAs' own lists; prompt sets that begin and end on and off the 32-key blocks of a thread
    wl = S.Workload(name="xiwalk", config_id=134, batch=4, tiles=((64, 32),), n_text=130, hidden=64, n_q_heads=8,
                    n_kv_heads=4, head_dim=head_dim, n_layers=16, layers=(3,), windows=(8,), keep=(0.5,))
    assert 16 * wl.n_q_heads * wl.batch > 3 * _sm_count()
    plan = H.make_plan(wl)
    inp = H.prepare_stage(wl, 0)
    late = wl.n_text + 700
    inp["k"][:, 1, late] *= 256.0                              # a power of two: still bf16 values
    gpu = H.gpu_stage(plan, wl, 0, inp, want_lse=True, text_ranges=text_ranges)
    del gpu["k_out"], gpu["v_out"]      # the scaled key row is outside the value range the bf16 K/V tolerance is meant for
    sub = {k: (v[[2]] if isinstance(v, np.ndarray) and v.shape[:1] == (4,) else v) for k, v in inp.items()}
    H.compare_stage(wl, 0, inp, H.oracle_stage(wl, 0, sub, text_ranges=text_ranges), gpu, samples=[2])
    H.check_lse_out(inp, gpu, wl.n_q_heads, wl.n_kv_heads, [2], atol=4e-2)
    plan.close()


def test_cfg2_lse_mode_full_size_sampled():
    # the benchmark shape in ATTN_LSE mode (5888 work items walked by 2 CTAs per SM), bench.py's streams; the
    # log-sum-exp input comes from plain torch ops, the oracle derives xi from Q and K alone
    stats = H.run_schedule(S.workload("cfg2"), xi_mode="lse", lse_source="torch", oracle_samples=[0, 5],
                           **_bench_streams())
    assert [s["n_out"] for s in stats] == [[1440] * 8, [720] * 8, [360] * 8]


@pytest.mark.parametrize("hidden,ragged", [(64, False), (72, True)])
def test_fd_persistent_ctas_take_several_tiles(hidden, ragged):
    # 160 samples x 36 windows of 16 tokens: 5760 CTAs of the streaming FD kernel, a window each, in many waves, with
    # hidden sizes of one and two chunks a row; the ragged variant gives every sample its own subset of the grid under
    # a plan built for subsets.  (CTAs of the tiled kernel that take several tiles: see
    # test_fd_tiles_of_a_window_larger_than_the_plan_expects.)
    wl = S.Workload(name="fdmulti", config_id=131, batch=160, tiles=((24, 24),), n_text=4, hidden=hidden,
                    n_q_heads=2, n_kv_heads=1, head_dim=64, n_layers=16, layers=(3,), windows=(6,), keep=(0.5,))
    first = None
    if ragged:
        rng = np.random.default_rng(77)
        full = np.arange(wl.n_vis, dtype=np.int32)
        first = [np.sort(rng.choice(full, int(rng.integers(500, 577)), replace=False)).astype(np.int32)
                 for _ in range(wl.batch)]
    stats = H.run_schedule(wl, xi_mode="uniform", oracle_samples=[0, 17, 159], ragged=ragged, first_pos=first)
    info = stats[0]["info"]
    assert info.uses_tensor_cores == 1 and info.fd_tiles * wl.batch > 2 * _sm_count()


@pytest.mark.parametrize("hidden", [72, 776])
@pytest.mark.parametrize("grid", [(3, 3), (4, 4), (3, 6), (4, 8), (3, 11), (6, 8), (7, 7), (8, 8), (5, 13), (8, 10), (9, 9)])
def test_fd_windows_around_groups_of_eight_nodes(grid, hidden):
    # one window of rows x cols tokens: the larger side just below, at and above the 8, 16, 24, 32 and 40 nodes the
    # streaming FD kernel's variants hold (41: the tcgen05 kernel); hidden sizes that end inside a chunk of columns
    wl = S.Workload(name="fdside", config_id=132, batch=3, tiles=(grid,), n_text=4, hidden=hidden, n_q_heads=2,
                    n_kv_heads=1, head_dim=64, n_layers=16, layers=(3,), windows=(1,), keep=(0.6,))
    H.run_schedule(wl, xi_mode="uniform")
    H.run_schedule(dataclasses.replace(wl, batch=1), xi_mode="uniform", direction="b2a", metric="l2")


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("grid", [(3, 5), (4, 4), (3, 6), (4, 8), (3, 11), (6, 8), (8, 8), (8, 10)])
def test_fd_narrow_rows_of_many_windows(grid, dtype):
    # more windows than SMs and rows of at most 1.5 KB: CTAs of two warps, at the edges of every variant's 8 to 40 nodes a side
    wl = S.Workload(name="fdnarrow", config_id=145, batch=151, tiles=(grid,), n_text=4, hidden=72, n_q_heads=2,
                    n_kv_heads=1, head_dim=64, n_layers=16, layers=(3,), windows=(1,), keep=(0.6,))
    H.run_schedule(wl, dtype=dtype, xi_mode="uniform", oracle_samples=[0, 75, 150])


@pytest.mark.parametrize("grid,windows,seed", [((12, 20), (5, 3), 282), ((12, 32), (3, 2), 4)])
def test_fd_window_larger_than_the_plan_expects(grid, windows, seed):
    # a near-full subset of the grid moves tokens between windows: one window of the second stage has a node more a
    # side than any window of the full grid (8, 24), so the streaming FD kernel walks it in blocks
    wl = S.Workload(name="fdwalk", config_id=133, batch=2, tiles=(grid,), n_text=4, hidden=776, n_q_heads=2,
                    n_kv_heads=1, head_dim=64, n_layers=16, layers=(3, 7), windows=windows, keep=(0.5, 0.5))
    rng = np.random.default_rng(seed)
    full = np.arange(grid[0] * grid[1], dtype=np.int32)
    missing = int(rng.integers(4, 14))
    subset = np.sort(rng.choice(full, full.size - missing, replace=False)).astype(np.int32)
    H.run_schedule(wl, xi_mode="given", first_pos=[subset, full])


@pytest.mark.parametrize("batch,hidden", [(2, 776), (30, 72), (45, 72)])
def test_fd_tiles_of_a_window_larger_than_the_plan_expects(batch, hidden):
    # the second stage's windows of up to 272 tokens are expected three quarters full (one tile of 128 x 128 nodes); here
    # some are full (136 a side), so a CTA takes four tiles in a row: ring phases, accumulator barrier and lists run on.
    # 8, 120 and 180 tiles: clusters, the deep ring, and neither
    wl = S.Workload(name="tilewalk", config_id=137, batch=batch, tiles=((32, 34),), n_text=4, hidden=hidden, n_q_heads=2,
                    n_kv_heads=1, head_dim=64, n_layers=16, layers=(3, 7), windows=(1, 2), keep=(0.75, 0.6))
    rows, cols = np.divmod(np.arange(wl.n_vis, dtype=np.int32), 34)
    window = (rows >= 16) * 2 + (cols >= 17)
    three = np.nonzero(window != 2)[0].astype(np.int32)
    one = np.concatenate([np.nonzero(window == 1)[0], np.nonzero(window != 1)[0][::5]])
    pos = [three if b % 2 == 0 else np.sort(one).astype(np.int32) for b in range(batch)]
    H.run_schedule(wl, xi_mode="uniform", stages=[1], ragged=True, first_pos=pos, oracle_samples=[0, 1, batch - 1])


@pytest.mark.parametrize("grid,w", [((32, 32), 5), ((25, 41), 4), ((32, 64), 8), ((45, 46), 7), ((64, 64), 11),
                                    ((64, 65), 9), ((90, 91), 16), ((91, 91), 12), ((96, 100), 12)])
def test_map_of_streaming_windows_over_cluster_sizes(grid, w):
    # samples at the borders between one, two, four and eight CTAs and between one and two tokens per thread of the
    # map kernel, one sample with the full grid and one with a subset of it (the cut between CTAs then falls elsewhere)
    wl = S.Workload(name="mapcs", config_id=135, batch=2, tiles=(grid,), n_text=5, hidden=64, n_q_heads=2,
                    n_kv_heads=1, head_dim=64, n_layers=16, layers=(3,), windows=(w,), keep=(0.57,))
    full = np.arange(wl.n_vis, dtype=np.int32)
    subset = np.sort(np.random.default_rng(w).choice(full, wl.n_vis * 5 // 7, replace=False)).astype(np.int32)
    H.run_schedule(wl, xi_mode="given", ragged=True, first_pos=[full, subset])


@pytest.mark.parametrize("grid,w,batch,hidden", [
    ((9, 9), 1, 120, 72),       # 41 nodes a side, a tile per SM: the deep ring
    ((16, 16), 1, 1, 776),      # 128 a side, clusters of eight
    ((16, 16), 1, 160, 72),     # 128 a side, more tiles than SMs, no cluster
    ((7, 37), 1, 2, 328),       # 130 and 129 a side: tiles of one and two rows
    ((33, 62), 2, 1, 200),      # windows of 496 to 527 tokens
    ((66, 62), 1, 1, 72),       # one window of 4092 tokens: the most the lists of a CTA hold
    ((70, 64), 1, 1, 72),       # one of 4480: window lists and keys through atomics
])
def test_fd_tiles_over_window_sizes(grid, w, batch, hidden):
    wl = S.Workload(name="fdtile", config_id=136, batch=batch, tiles=(grid,), n_text=4, hidden=hidden, n_q_heads=2,
                    n_kv_heads=1, head_dim=64, n_layers=16, layers=(3,), windows=(w,), keep=(0.6,))
    samples = sorted({0, batch // 2, batch - 1})
    H.run_schedule(wl, xi_mode="uniform", oracle_samples=samples)
    if batch < 10 and grid[0] * grid[1] < 3000:
        H.run_schedule(wl, xi_mode="uniform", direction="b2a", metric="l2sq", oracle_samples=samples)


# ---- subsets of the grid: capacities ---------------------------------------------------------------------------

@pytest.mark.parametrize("grid,hidden", [((8, 8), 1024), ((12, 16), 256), ((12, 16), 768), ((12, 16), 1024),
                                         ((13, 17), 2056), ((16, 32), 4096)])
def test_repeated_source_rows_merge_by_index(grid, hidden):
    """Every source row of the one window is the same, so all of them have the same lowest score bit for bit and only the
    tie rule decides: the lowest source indices go, into one destination.  Few windows: the FD kernel splits the hidden
    dimension over clusters of 2, 4 or 8 CTAs (256 / 768 / 1024 channels and more) that each finish some of the rows."""
    import torch
    import paper_2605_00789_b200 as L
    wl = S.Workload(name="ties", config_id=131, batch=1, tiles=(grid,), n_text=5, hidden=hidden, n_q_heads=2,
                    n_kv_heads=2, head_dim=64, n_layers=4, layers=(2,), windows=(1,), keep=(0.75,))
    n = grid[0] * grid[1]
    plan = H.make_plan(wl, xi_mode="uniform")
    gen = torch.Generator(device="cuda")
    for seed in range(3):
        gen.manual_seed(seed)
        src = torch.randn((hidden,), generator=gen, device="cuda")
        hidden_in = torch.randn((1, wl.n_text + n, hidden), generator=gen, device="cuda")
        vis = hidden_in[:, wl.n_text:]
        vis.mul_(0.3).add_(src)                      # destinations near the source: scores far from 1, with all their digits
        vis[:, 0::2] = src
        out = L.StageBuffers(plan, 0, wl.n_text + plan.stage_info(0).cap_out, "cuda")
        L.compress_layer(plan, 0, hidden_in.bfloat16(), out, vis_begin=wl.n_text)
        removed = n - int(np.ceil(0.75 * n))
        assert int(out.status) == 0 and int(out.n_vis_out) == n - removed
        dst = out.dst[0].cpu().numpy()
        left = np.ones(n, dtype=bool)
        left[0:2 * removed:2] = False                # the first `removed` sources
        np.testing.assert_array_equal(out.pos_out[0, :n - removed].cpu().numpy(), np.nonzero(left)[0])
        assert len(set(dst[0:2 * removed:2])) == 1
    plan.close()


def _near_full_subset():
    """576-token grid, windows 6 / 4 / 2 (not nested): a sample that misses 8 positions reaches the second stage
    with 146 A nodes, two more than the full grid's 144 (found with the oracle, seed fixed)."""
    wl = dataclasses.replace(S.workload("cfg1r"), batch=2, hidden=64, n_q_heads=2, n_kv_heads=2, head_dim=64, n_text=8)
    rng = np.random.default_rng(9000)
    full = np.arange(576, dtype=np.int32)
    n_missing = int(rng.integers(1, 12))
    subset = np.sort(rng.choice(full, 576 - n_missing, replace=False)).astype(np.int32)
    return wl, [subset, full]


def test_near_full_subset_through_two_stages_under_a_ragged_plan():
    wl, first = _near_full_subset()
    stats = H.run_schedule(wl, stages=[0, 1], ragged=True, first_pos=first)
    assert stats[1]["info"].cap_a >= 146 and stats[1]["info"].counts_exact == 0


def test_subset_given_to_a_full_grid_plan_raises_the_count_bit():
    """The same subset under a plan built for full grids: at the second stage it has more A nodes than the plan
    holds.  The sample then passes through unmerged (cut at cap_out), the COUNT bit is raised, nothing is written
    out of a row, and the full-grid sample beside it still matches the oracle."""
    wl, first = _near_full_subset()
    plan = H.make_plan(wl, batch=2)
    inp0 = H.prepare_stage(wl, 0, first)
    g0 = H.gpu_stage(plan, wl, 0, inp0)
    H.compare_stage(wl, 0, inp0, H.oracle_stage(wl, 0, inp0), g0)           # stage 0 holds any subset
    pos1 = [g0["pos_out"][b, :int(g0["n_vis_out"][b])] for b in range(2)]
    info = plan.stage_info(1)
    assert info.cap_a == 144 and info.cap_out == 144
    inp1 = H.prepare_stage(wl, 1, pos1)
    g1 = H.gpu_stage(plan, wl, 1, inp1)
    assert int(g1["status"][0]) == 8
    sub = {k: (v[[1]] if isinstance(v, np.ndarray) and v.shape[:1] == (2,) else v) for k, v in inp1.items()}
    H.compare_stage(wl, 1, inp1, H.oracle_stage(wl, 1, sub), g1, samples=[1], expect_status=8)
    vb = inp1["vis_begin"]
    assert int(g1["n_vis_out"][0]) == info.cap_out
    np.testing.assert_array_equal(g1["pos_out"][0, :144], pos1[0][:144])
    np.testing.assert_array_equal(g1["hidden_out"][0, vb:vb + 144], inp1["hidden"][0, vb:vb + 144])
    plan.close()


# ---- xi summed over the heads, and weights: with the merge of the rows, or in front of it -------------------------

def _layer_in_form(plan, form, rows, nt, **kw):
    """Stage 0 in one of the forms that make the weights: "merge" (with the merge of the rows), "map" (a map behind xi, for a
    caller that waits for the map of a short launch of few heads or tokens), "kernel" (weights_kernel: the launch is long, by
    rows behind the vision block), "kernel and event" (the same where the caller waits for the map) or "event" (weights_kernel in
    a short launch of many heads and tokens, for a caller that waits).  The launches of the call show that it was the form."""
    import torch
    import bench
    import paper_2605_00789_b200 as L
    after = 0
    if "kernel" in form:
        after = (24 << 20) // (rows.shape[0] * rows.shape[2] * rows.element_size())
        rows = torch.cat([rows, torch.zeros((rows.shape[0], after, rows.shape[2]), device="cuda", dtype=rows.dtype)], 1)
    if form in ("map", "event", "kernel and event"):
        kw["map_event"] = torch.cuda.Event()
        kw["map_event"].record()
    out = L.StageBuffers(plan, 0, nt + plan.stage_info(0).cap_out + after)
    out.workspace.fill_(255)                           # (a sum over heads that were not written is not a number)
    call = lambda: L.compress_layer(plan, 0, rows, out, vis_begin=nt, n_text_after=after, **kw)
    call()
    torch.cuda.synchronize()
    assert bench.count_launches(call) == (4 if form in ("merge", "map") else 5)
    return out


MAP_OUTPUTS = ("n_vis_out", "pos_out", "dst", "grp_off", "grp_src", "xi_out", "weight")


@pytest.mark.parametrize("heads,dtype", [(1, "bf16"), (6, "fp32"), (7, "bf16"), (28, "bf16"), (32, "bf16"), (33, "bf16"),
                                         (40, "bf16"), (64, "bf16"), (70, "fp32"), (100, "bf16")])
@pytest.mark.parametrize("xi_mode", ["attn", "lse"])
def test_xi_and_weights_have_the_same_bits_in_every_form(heads, dtype, xi_mode):
    """The heads of a token are added in one order, whichever kernel adds them: with the merge, in the map, in a kernel of their
    own, and for a sample alone (32 heads to a round, a round that is not full, two and four rounds)."""
    import torch
    import paper_2605_00789_b200 as L
    b, nt, tiles = 3, 9, [(13, 17), (9, 11)]
    n = sum(r * c for r, c in tiles)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    plan = lambda batch, h=heads: L.Plan(batch, 72, h, 1, 64, 8, tiles, [2], [3], [0.6], 70000, ragged_input=True,
                                dtype=L.BF16 if dtype == "bf16" else L.FP32,
                                xi_mode=L.XI_ATTN_FULL if xi_mode == "attn" else L.XI_ATTN_LSE)
    gen = torch.Generator(device="cuda").manual_seed(heads)
    rows = torch.randn((b, nt + n, 72), generator=gen, device="cuda").to(dt)
    q, k = (torch.randn((b, h, nt + n, 64), generator=gen, device="cuda").to(dt) for h in (heads, 1))
    pos = torch.full((b, n), -1, device="cuda", dtype=torch.int32)
    counts = [n, 131, 5]
    for i, m in enumerate(counts):
        pos[i, :m] = torch.randperm(n, generator=gen, device="cuda")[:m].sort().values.int()
    kw = dict(q=q, k=k, pos=pos, n_vis=torch.tensor(counts, device="cuda", dtype=torch.int32))
    if xi_mode == "lse":
        kw["lse"] = 3.0 + torch.rand((b, heads, nt + n), generator=gen, device="cuda")
    waits = "event" if xi_mode == "attn" and heads > 16 else "map"      # 960 tokens
    found = {form: _layer_in_form(plan(b), form, rows, nt, **kw) for form in ("merge", waits, "kernel", "kernel and event")}
    want = found["merge"]
    assert int(want.status) == 0 and bool((want.xi_out[0] > 0).all())
    for form, out in found.items():
        for name in MAP_OUTPUTS:
            assert torch.equal(getattr(out, name), getattr(want, name)), (form, name)
        for i in range(b):
            end = nt + int(want.n_vis_out[i])
            assert torch.equal(out.hidden_out[i, :end], want.hidden_out[i, :end]), form
    for i in range(b if dtype == "bf16" else 0):       # (the fp32 xi kernel cuts a row's keys by the size of the launch)
        alone = _layer_in_form(plan(1), "merge", rows[i:i + 1], nt, **{key: t[i:i + 1] for key, t in kw.items()})
        for name in ("xi_out", "weight"):
            assert torch.equal(getattr(alone, name)[0, :counts[i]], getattr(want, name)[i, :counts[i]]), (i, name)
    # against the sum in double precision of what a call for each head reports
    if heads in (7, 33):
        one = plan(b, 1)
        total = torch.zeros((b, n), device="cuda", dtype=torch.float64)
        for h in range(heads):
            more = dict(kw, q=q[:, h:h + 1])
            if xi_mode == "lse":
                more["lse"] = kw["lse"][:, h:h + 1].contiguous()
            total += _layer_in_form(one, "merge", rows, nt, **more).xi_out.double()
        torch.testing.assert_close(want.xi_out.double(), total, rtol=heads * 2.0 ** -24, atol=0)


@pytest.mark.parametrize("heads", [7, 32])
def test_xi_and_weights_have_the_same_bits_in_the_list_form(heads):
    """Eight windows of 64 x 64 tokens: their keys do not fit the built-in workspace beside the heads' sums, so that call takes
    the list form, whose selection adds the heads, too."""
    import torch
    import paper_2605_00789_b200 as L
    b, n, nt = 20 if heads == 7 else 8, 4096, 3
    plan = L.Plan(b, 64, heads, 1, 64, 8, [(64, 64)], [2], [1], [0.6], nt)
    assert plan.stage_info(0).workspace_bytes > L.BUILTIN_WS_BYTES
    gen = torch.Generator(device="cuda").manual_seed(heads)
    rows = torch.randn((b, nt + n, 64), generator=gen, device="cuda").bfloat16()
    q, k = (torch.randn((b, h, nt + n, 64), generator=gen, device="cuda").bfloat16() for h in (heads, 1))
    found = []
    for call in (L.compress_layer, L.compress_layer_builtin_ws):
        out = L.StageBuffers(plan, 0, nt + plan.stage_info(0).cap_out)
        call(plan, 0, rows, out, vis_begin=nt, q=q, k=k)
        torch.cuda.synchronize()
        found.append(out)
    for name in MAP_OUTPUTS:
        assert torch.equal(getattr(found[0], name), getattr(found[1], name)), name
    plan.close()


@pytest.mark.parametrize("heads", [1, 7, 33, 40, 70])
@pytest.mark.parametrize("before_merge", [False, True])
def test_weights_over_head_counts(heads, before_merge):
    """The heads are taken 32 at a time, in one and in two rounds: by the merge's warps and, with a map event, by the threads of
    a map behind xi or, beyond 16 heads, by weights_kernel.  (All give the same bits, see above.)"""
    import torch
    wl = S.Workload(name="heads", config_id=133, batch=3, tiles=((13, 17), (9, 11)), n_text=9, hidden=72, n_q_heads=heads,
                    n_kv_heads=1, head_dim=64, n_layers=8, layers=(2, 5), windows=(3, 2), keep=(0.6, 0.5))
    H.run_schedule(wl, kv_stream=torch.cuda.Stream() if before_merge else None)


@pytest.mark.parametrize("grid", [(11, 11), (13, 17), (32, 40)])
@pytest.mark.parametrize("form", ["merge", "map", "kernel"])
def test_weights_of_a_group_of_all_sources(grid, form):
    """Equal source rows all join one destination: groups of 61, 111 and 641 members, below and beyond what the kernels keep
    on chip.  The weights are the reported xi over their sum (single precision: 1e-5 over up to 641 terms), and the merged
    row is the weighted sum of the members' rows."""
    import torch
    wl = S.Workload(name="onegroup", config_id=134, batch=1, tiles=(grid,), n_text=5, hidden=1032, n_q_heads=6,
                    n_kv_heads=2, head_dim=64, n_layers=4, layers=(2,), windows=(1,), keep=(0.5,))
    n, na = grid[0] * grid[1], (grid[0] * grid[1] + 1) // 2
    removed = n - int(np.ceil(0.5 * n))
    plan = H.make_plan(wl, max_text=20000)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(grid[0])
    hidden_in = torch.randn((1, wl.n_text + n, wl.hidden), generator=gen, device="cuda")
    hidden_in[:, wl.n_text::2] = hidden_in[:, wl.n_text:wl.n_text + 1].clone()
    hidden_in = hidden_in.bfloat16()
    q = torch.randn((1, 6, wl.n_text + n, 64), generator=gen, device="cuda").bfloat16()
    k = torch.randn((1, 2, wl.n_text + n, 64), generator=gen, device="cuda").bfloat16()
    out = _layer_in_form(plan, form, hidden_in, wl.n_text, q=q, k=k)
    assert int(out.status) == 0 and int(out.n_vis_out) == n - removed and na - removed in (0, 1)
    off, src = out.grp_off[0].cpu().numpy(), out.grp_src[0].cpu().numpy()
    xi, weight = (t[0].cpu().numpy().astype(np.float64) for t in (out.xi_out, out.weight))
    rows, merged = hidden_in[0].float().cpu().numpy(), out.hidden_out[0].float().cpu().numpy()
    sizes = np.diff(off[:n - removed + 1])
    assert (xi > 0).all() and sizes.max() == removed + 1 and sizes.sum() == n
    for o in (int(sizes.argmax()), int(sizes.argmin())):
        members = src[off[o]:off[o + 1]]
        np.testing.assert_allclose(weight[members], xi[members] / xi[members].sum(), rtol=1e-5, atol=0)
        want = weight[members] @ rows[wl.n_text + members]
        np.testing.assert_allclose(merged[wl.n_text + o], want, rtol=2 ** -8, atol=1e-4)
    plan.close()


@pytest.mark.parametrize("xi_mode,form", [("given", None), ("lse", "merge"), ("lse", "map"), ("lse", "kernel")])
def test_an_infinite_score_leaves_no_number(xi_mode, form):
    """xi / sum is inf / inf for a token whose score is infinite, alone or in a group: its weight and its row are NaN, and no
    other group's are.  (A log-sum-exp of -200 overflows the exponentials of its row.)"""
    import torch
    import paper_2605_00789_b200 as L
    n, nt = 144, 5
    plan = L.Plan(1, 264, 4, 4, 64, 4, [(12, 12)], [2], [3], [0.55], 60000, xi_mode=L.XI_GIVEN if xi_mode == "given" else L.XI_ATTN_LSE)
    gen = torch.Generator(device="cuda").manual_seed(11)
    rows = torch.randn((1, nt + n, 264), generator=gen, device="cuda").bfloat16()
    kw = {}
    if xi_mode == "given":
        kw["xi"] = 0.5 + torch.rand((1, n), generator=gen, device="cuda")
        kw["xi"][:, ::7] = float("inf")
        out = L.StageBuffers(plan, 0, nt + plan.stage_info(0).cap_out, "cuda")
        L.compress_layer(plan, 0, rows, out, vis_begin=nt, **kw)
    else:
        kw["q"], kw["k"] = (torch.randn((1, 4, nt + n, 64), generator=gen, device="cuda").bfloat16() for _ in range(2))
        kw["lse"] = torch.full((1, 4, nt + n), 3.0, device="cuda")
        kw["lse"][:, :, nt::7] = -200.0
        out = _layer_in_form(plan, form, rows, nt, **kw)
    inf = ~torch.isfinite(out.xi_out[0])
    assert torch.equal(inf.nonzero()[:, 0].cpu(), torch.arange(0, n, 7)) and bool((out.xi_out[0][inf] > 0).all())
    assert torch.equal(torch.isnan(out.weight[0]), inf)
    off, src = out.grp_off[0].cpu(), out.grp_src[0].cpu()
    kinds = set()
    for o in range(int(out.n_vis_out)):
        members = src[off[o]:off[o + 1]].long()
        bad = bool(inf.cpu()[members].any())
        assert torch.isnan(out.hidden_out[0, nt + o]).all() if bad else torch.isfinite(out.hidden_out[0, nt + o]).all()
        kinds.add((bad, len(members) > 1))
    assert len(kinds) == 4
    plan.close()


@pytest.mark.parametrize("form", ["merge", "map", "kernel"])
def test_xi_of_tokens_cut_at_the_capacity_is_reported(form):
    """A subset under a full-grid plan keeps all of its tokens and is cut at cap_out: those behind the cut belong to no group,
    and their xi is reported all the same -- the same as under a plan that has room for them."""
    import torch
    import bench
    wl, first = _near_full_subset()
    plan, roomy = H.make_plan(wl, batch=2, max_text=120000), H.make_plan(wl, batch=2, ragged=True)
    g0 = H.gpu_stage(plan, wl, 0, H.prepare_stage(wl, 0, first))
    pos1 = [g0["pos_out"][b, :int(g0["n_vis_out"][b])] for b in range(2)]
    inp1 = H.prepare_stage(wl, 1, pos1)
    whole = H.gpu_stage(roomy, wl, 1, inp1)
    after, launches = 0, []
    if form == "kernel":                               # a long launch, by rows behind the vision block
        after = (24 << 20) // (2 * wl.hidden * 2)
        inp1["hidden"] = np.pad(inp1["hidden"], ((0, 0), (0, after - 1), (0, 0)))
        del inp1["v"]

    def layer(*args, **kw):
        import paper_2605_00789_b200 as L
        launches.append(bench.count_launches(lambda: L.compress_layer(*args, **kw)))
        L.compress_layer(*args, **kw)

    cut = H.gpu_stage(plan, wl, 1, inp1, n_text_after=after, kv_stream=torch.cuda.Stream() if form == "map" else None, layer_fn=layer)
    assert launches == [5 if form == "kernel" else 4]
    n = int(inp1["n_vis"][0])
    assert int(cut["status"][0]) == 8 and int(cut["n_vis_out"][0]) < n
    np.testing.assert_array_equal(cut["xi_out"][0, :n] > 0, True)
    np.testing.assert_allclose(cut["xi_out"][0, :n], whole["xi_out"][0, :n], rtol=1e-6, atol=0)
    plan.close()
    roomy.close()


@pytest.mark.parametrize("xi_mode,dtype", [("attn", "bf16"), ("lse", "bf16"), ("attn", "fp32")])
@pytest.mark.parametrize("streams", [1, 2])
@pytest.mark.parametrize("hidden", [64, 2048])
def test_counts_replaced_in_place(xi_mode, dtype, streams, hidden):
    """One array for the counts that come in and those that go out gives what two arrays give, with more work items of xi than
    CTAs and little else to do (hidden 64), and where the weights have a kernel of their own otherwise (2048: 28 MB)."""
    import torch
    import paper_2605_00789_b200 as L
    b, grid, nt, h, dh = 12, (31, 37), 7, 12, 64
    n = grid[0] * grid[1]
    xm = L.XI_ATTN_FULL if xi_mode == "attn" else L.XI_ATTN_LSE
    plan = L.Plan(b, hidden, h, 4, dh, 8, [grid], [3], [5], [0.5], nt, xi_mode=xm, ragged_input=True,
                  dtype=L.BF16 if dtype == "bf16" else L.FP32)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(5)
    rows = torch.randn((b, nt + n, hidden), generator=gen, device="cuda").to(dt)
    q, k = (torch.randn((b, heads, nt + n, dh), generator=gen, device="cuda").to(dt) for heads in (h, 4))
    pos = torch.full((b, n), -1, device="cuda", dtype=torch.int32)
    counts = [n - 97 * (i % 5) for i in range(b)]
    for i, m in enumerate(counts):
        pos[i, :m] = torch.randperm(n, generator=gen, device="cuda")[:m].sort().values.int()
    kw = dict(vis_begin=nt, q=q, k=k, pos=pos)
    if xi_mode == "lse":
        kw["lse"] = 3.0 + torch.rand((b, h, nt + n), generator=gen, device="cuda")
    if streams == 2:
        kw["aux_stream"] = torch.cuda.Stream()
    found = []
    for in_place in (False, True):
        n_vis = torch.tensor(counts, device="cuda", dtype=torch.int32)
        out = L.StageBuffers(plan, 0, nt + plan.stage_info(0).cap_out)
        out.hidden_out.zero_()
        out.workspace.fill_(255)                       # (a sum over heads that were not written is not a number)
        if in_place:
            out.n_vis_out = n_vis
        L.compress_layer(plan, 0, rows, out, n_vis=n_vis, **kw)
        found.append(out)
    two, one = found
    assert int(two.status) == int(one.status) == 0 and int(one.n_vis_out.max()) < min(counts)
    for name in MAP_OUTPUTS + ("hidden_out",):
        assert torch.equal(getattr(two, name), getattr(one, name)), name
    plan.close()


# ---- seeded random geometries ---------------------------------------------------------------------

def _random_workload(seed):
    """Tiles, windows, keep ratios, head layout and sizes drawn from a seeded generator: ragged windows, several
    tiles per sample, 600 to 4500 tokens (one to eight CTAs per sample in the selection kernel), hidden sizes
    that are and are not multiples of 64, head sizes with and without a tensor-core path."""
    rng = np.random.default_rng(7000 + seed)
    n_tiles = int(rng.integers(1, 4))
    big = seed % 3 == 0
    tiles = tuple((int(rng.integers(18, 50 if big else 30)), int(rng.integers(18, 46 if big else 26)))
                  for _ in range(n_tiles))
    smallest = min(min(t) for t in tiles)
    windows = tuple(sorted((int(rng.integers(1, min(7, smallest // 2))) for _ in range(3)), reverse=True))
    n_kv = int(rng.choice([1, 2, 4]))
    return S.Workload(name=f"rand{seed}", config_id=100 + seed, batch=int(rng.integers(1, 4)), tiles=tiles,
                      n_text=int(rng.integers(1, 180)), hidden=int(rng.choice([64, 72, 192, 320, 520])),
                      n_q_heads=n_kv * int(rng.choice([1, 2])), n_kv_heads=n_kv,
                      head_dim=int(rng.choice([64, 128, 128, 32])), n_layers=16, layers=(3, 7, 11),
                      windows=windows, keep=tuple(float(k) for k in rng.uniform(0.5, 0.9, size=3).round(2)))


@pytest.mark.parametrize("seed", range(16))
def test_random_geometry(seed):
    wl = _random_workload(seed)
    # K/V side: merge or gather, contiguous or paged caches (pages of 16 or 5 tokens), both cache layouts
    H.run_schedule(wl, xi_mode=["attn", "given", "lse"][seed % 3], dtype="fp32" if seed == 4 else "bf16",
                   engine="simt" if seed == 4 else "auto", kv_mode=["merge", "gather"][(seed // 2) % 2],
                   paged=[0, 16, 0, 5][seed % 4], kv_layout="bnhd" if seed % 4 == 2 else "bhnd")


def test_selection_over_eight_ctas_ragged_windows():
    # 4480 tokens per sample (a cluster of eight CTAs in the selection kernel), windows that do not divide
    # the grid, a single large window at the last stage (1344 tokens: the per-window rank loops at length)
    wl = S.Workload(name="sel8", config_id=120, batch=2, tiles=((70, 64),), n_text=9, hidden=64, n_q_heads=2,
                    n_kv_heads=1, head_dim=64, n_layers=16, layers=(3, 7, 11), windows=(6, 3, 1),
                    keep=(0.6, 0.5, 0.7))
    stats = H.run_schedule(wl, xi_mode="given")
    assert stats[0]["n_out"][0] < 4480 * 0.6 + 40


@pytest.mark.parametrize("engine", ["simt", "auto"])
def test_windows_of_one_and_two_tokens(engine):
    # a 6 x 8 grid cut 6 x 6: windows of one token (no B node: nothing to merge) and of two (one A, one B);
    # then 3 x 3 and a single window over what is left
    wl = S.Workload(name="w12", config_id=122, batch=2, tiles=((6, 8),), n_text=3, hidden=64, n_q_heads=2,
                    n_kv_heads=1, head_dim=64, n_layers=16, layers=(3, 7, 11), windows=(6, 3, 1),
                    keep=(0.5, 0.6, 0.5))
    stats = H.run_schedule(wl, engine=engine)
    assert stats[0]["n_out"] == [36, 36]          # twelve two-token windows lose one token each


def test_selection_with_several_tokens_per_thread():
    # 9600 tokens per sample: more than the 8 x 1024 threads of the largest cluster, so every phase of the
    # selection kernel loops and its prefix sums take the two-pass path
    wl = S.Workload(name="sel9600", config_id=121, batch=1, tiles=((100, 96),), n_text=7, hidden=64, n_q_heads=2,
                    n_kv_heads=2, head_dim=64, n_layers=16, layers=(3, 7, 11), windows=(6, 3, 2),
                    keep=(0.6, 0.5, 0.7))
    H.run_schedule(wl, xi_mode="given", stages=[0, 1])


# ---- full benchmark shapes, compared on the samples the oracle can finish in seconds -----------------

def _bench_streams():
    # the schedule bench.py times: second stream inside the call (window build and FD beside xi), K/V
    # compaction on a third stream behind the map event
    import torch
    return dict(aux_stream=torch.cuda.Stream(), kv_stream=torch.cuda.Stream())


def test_cfg2_full_size_sampled():
    stats = H.run_schedule(S.workload("cfg2"), oracle_samples=[0, 5], **_bench_streams())
    assert [s["n_out"] for s in stats] == [[1440] * 8, [720] * 8, [360] * 8]


def test_cfg2_full_size_one_stream():
    H.run_schedule(S.workload("cfg2"), oracle_samples=[3], stages=[0])


def test_cfg3_full_schedule_sampled():
    stats = H.run_schedule(S.workload("cfg3"), oracle_samples=[0, 31], **_bench_streams())
    assert [s["n_out"] for s in stats] == [[288] * 32, [144] * 32, [72] * 32]


def test_cfg4_gqa_video_full_schedule_sampled():
    # all three stages: later stages have few large tiles (128 x 128 entries), which the FD kernel splits
    # over clusters of CTAs, and 8192 -> 2048 tokens per sample for the clustered selection kernel
    stats = H.run_schedule(S.workload("cfg4"), oracle_samples=[1], **_bench_streams())
    assert [s["n_out"] for s in stats] == [[4096] * 2, [2048] * 2, [1024] * 2]


def test_cfg4g_large_windows_uniform_xi():
    # windows of 512, 1024 and 2048 tokens: FD tiles of 128 x 128 nodes whose keys the map kernel combines across the
    # blocks of destinations, and its selection among up to 1024 sources
    H.run_schedule(S.workload("cfg4g"), xi_mode="uniform", oracle_samples=[0])


@pytest.mark.parametrize("in_place", [False, True])
def test_heads_of_one_piece(in_place):
    # head_dim 8 in bf16: a head's row is a single 16-byte piece
    wl = S.Workload(name="piece", config_id=142, batch=2, tiles=((9, 7),), n_text=3, hidden=64, n_q_heads=4,
                    n_kv_heads=4, head_dim=8, n_layers=16, layers=(3,), windows=(2,), keep=(0.55,))
    H.run_schedule(wl, xi_mode="given", kv_in_place=in_place)


@pytest.mark.parametrize("batch,grid,in_place", [(40, (9, 7), False), (40, (9, 7), True), (1, (66, 70), True)])
def test_heads_of_one_piece_over_variants(batch, grid, in_place):
    # the form for many rows, and planes of one and of two CTAs per SM
    wl = S.Workload(name="pieces", config_id=146, batch=batch, tiles=(grid,), n_text=3, hidden=64, n_q_heads=4,
                    n_kv_heads=4, head_dim=8, n_layers=16, layers=(3,), windows=(6,), keep=(0.55,))
    H.run_schedule(wl, xi_mode="given", kv_in_place=in_place, oracle_samples=sorted({0, batch - 1}))


def test_weights_of_samples_with_a_token_per_cta():
    # at most eight tokens a sample: the map behind xi (the caller waits for the map alone) against the oracle, and
    # weights_kernel, whose clusters then have CTAs without a token, against it
    import torch
    wl = S.Workload(name="few", config_id=143, batch=3, tiles=((2, 4),), n_text=9, hidden=64, n_q_heads=4,
                    n_kv_heads=4, head_dim=64, n_layers=16, layers=(3,), windows=(1,), keep=(0.5,))
    H.run_schedule(wl, kv_stream=torch.cuda.Stream())
    gen = torch.Generator(device="cuda").manual_seed(3)
    for grid in ((1, 2), (2, 4), (3, 3), (2, 8), (1, 17)):
        few = dataclasses.replace(wl, tiles=(grid,))
        plan = H.make_plan(few, max_text=70000)
        n = 9 + grid[0] * grid[1]
        rows = torch.randn((3, n, 64), generator=gen, device="cuda").bfloat16()
        q, k = (torch.randn((3, 4, n, 64), generator=gen, device="cuda").bfloat16() for _ in range(2))
        short, long = (_layer_in_form(plan, form, rows, 9, q=q, k=k) for form in ("map", "kernel"))
        for name in MAP_OUTPUTS:
            assert torch.equal(getattr(short, name), getattr(long, name)), (grid, name)
        plan.close()


@pytest.mark.parametrize("grid,n_kv,head_dim,page,vb,after", [
    ((9, 7), 2, 8, 1, 0, 0),           # pages of one row (their index is divided, not multiplied)
    ((24, 24), 2, 24, 7, 13, 5),       # rows of three pieces, the first page begins in front of the vision block
    ((24, 24), 3, 128, 48, 47, 1),
    ((48, 48), 2, 128, 16, 5, 40),     # one CTA per SM
    ((24, 24), 2, 64, 70000, 3, 2),    # a page longer than the multiplier's range
])
@pytest.mark.parametrize("dtype,mode", [("bf16", "merge"), ("fp32", "merge"), ("bf16", "gather")])
def test_in_place_pages_equal_contiguous_bit_for_bit(grid, n_kv, head_dim, page, vb, after, dtype, mode):
    import torch
    import paper_2605_00789_b200 as L
    b, n = 2, grid[0] * grid[1]
    plan = L.Plan(b, 64, n_kv, n_kv, head_dim, 8, [grid], [3], [2], [0.55], vb + after,
                  dtype=L.BF16 if dtype == "bf16" else L.FP32, xi_mode=L.XI_GIVEN)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(7)
    rows = vb + n + after
    hidden = torch.randn((b, rows, 64), generator=gen, device="cuda").to(dt)
    out = L.StageBuffers(plan, 0, vb + plan.stage_info(0).cap_out + after)
    L.compress_layer(plan, 0, hidden, out, vis_begin=vb, n_text_after=after,
                     xi=torch.rand((b, n), generator=gen, device="cuda") + 0.1)
    m = L.KV_MERGE if mode == "merge" else L.KV_GATHER
    k, v = (torch.randn((b, n_kv, rows, head_dim), generator=gen, device="cuda").to(dt) for _ in range(2))
    kd, vd = torch.zeros_like(k), torch.zeros_like(v)
    L.compact_kv(plan, 0, out, k, v, kd, vd, vis_begin=vb, n_text_after=after, mode=m)
    blocks = -(-rows // page)
    table = torch.randperm(b * blocks, generator=gen, device="cuda").view(b, blocks).int()

    def pool(x):
        full = torch.zeros((b, n_kv, blocks * page, head_dim), device="cuda", dtype=dt)
        full[:, :, :rows] = x
        p = torch.empty((b * blocks, n_kv, page, head_dim), device="cuda", dtype=dt)
        p[table.reshape(-1).long()] = full.view(b, n_kv, blocks, page, head_dim).transpose(1, 2).reshape(p.shape)
        return p

    kp, vp = pool(k), pool(v)
    L.compact_kv(plan, 0, out, kp, vp, kp, vp, vis_begin=vb, n_text_after=after, mode=m, page_size=page,
                 src_block_table=table, dst_block_table=table)
    L.compact_kv(plan, 0, out, k, v, k, v, vis_begin=vb, n_text_after=after, mode=m)
    counts = out.n_vis_out.tolist()
    for want, paged, flat in ((kd, kp, k), (vd, vp, v)):
        got = paged[table.reshape(-1).long()].view(b, blocks, n_kv, page, head_dim).transpose(1, 2).reshape(b, n_kv, -1, head_dim)
        for i in range(b):
            end = vb + counts[i] + after
            assert torch.equal(got[i, :, :end], want[i, :, :end])
            assert torch.equal(flat[i, :, :end], want[i, :, :end])
    plan.close()


@pytest.mark.parametrize("grid,windows,batch", [((64, 64), 1, 1), ((48, 48), 2, 2), ((24, 24), 2, 1), ((256, 32), 4, 2)])
def test_scores_near_the_ends_of_the_norms_range(grid, windows, batch):
    # rows scaled by a power of two have the same cosines bit for bit; the tiled FD kernel compares them without a division
    # where all norms of a tile are between 1e-15 and 1e15, with and without clusters, and pair by pair elsewhere
    import torch
    import paper_2605_00789_b200 as L
    n = grid[0] * grid[1]
    plan = L.Plan(batch, 256, 2, 2, 64, 8, [grid], [3], [windows], [0.6], 4, xi_mode=L.XI_UNIFORM)
    gen = torch.Generator(device="cuda").manual_seed(11)
    rows = torch.randn((batch, 4 + n, 256), generator=gen, device="cuda").to(torch.bfloat16)
    rows[:, 4 + 7] = 0
    mixed = torch.ones((4 + n, 1), device="cuda")
    mixed[4 + 13::57] = 2.0 ** -60
    found = []
    for scale in (1.0, 2.0 ** -60, 2.0 ** 52, mixed):
        out = L.StageBuffers(plan, 0, 4 + plan.stage_info(0).cap_out)
        L.compress_layer(plan, 0, (rows.float() * scale).to(torch.bfloat16), out, vis_begin=4)
        found.append(out.dst.cpu())
    for other in found[1:]:
        assert torch.equal(found[0], other)
    plan.close()


@pytest.mark.parametrize("grid", [(1, 255), (1, 257), (1, 259), (3, 401), (1, 2049)])
@pytest.mark.parametrize("direction", ["a2b", "b2a"])
def test_selection_over_eighths_of_the_sources(grid, direction):
    # one window; up to 128 sources are walked by their own threads, more by eight warps in turns of 32
    wl = S.Workload(name="eighths", config_id=144, batch=1, tiles=(grid,), n_text=3, hidden=64, n_q_heads=2,
                    n_kv_heads=2, head_dim=64, n_layers=16, layers=(3,), windows=(1,), keep=(0.6,))
    H.run_schedule(wl, xi_mode="given", direction=direction)
