"""GPU parity: the CUDA library, called through its C ABI, against the fp64 CPU oracle on the same
seeded inputs.  Integer results (kept indices given identical scores, compacted rows) must be
bit-exact; salience scores within 2e-3 relative (bf16 inputs, fp32 accumulate)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_09244_b200 import mvla
from paper_2604_09244_b200 import workloads as W
from parity_util import (SALIENCE_RTOL, assert_salience_close, check_compaction, check_kept_against_oracle,
                         check_stagewise_exact, device_tensors, diag_records, run_and_check_step)

pytestmark = pytest.mark.gpu


# ------------------------------------------------------------------ compaction
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_compact_bit_exact_ragged(dtype):
    wl = W.small_workload(21, batch=3, D=264 if dtype == "bf16" else 260, H=3, d=64, dtype=dtype,
                          n_txt=(5, 19, 1), n_2d=(70, 130, 3), n_3d=(150, 37, 9))
    ctx = mvla.context_for(wl)
    dev = device_tensors(wl)
    rng = np.random.default_rng(0)
    kept, offs = [], [0]
    for s in wl.samples:
        k = np.sort(rng.choice(s.seq_len, size=int(rng.integers(1, s.seq_len + 1)), replace=False))
        kept.append(k.astype(np.int32))
        offs.append(offs[-1] + len(k))
    kept_d = torch.from_numpy(np.concatenate(kept)).cuda()
    offs_d = torch.tensor(offs, dtype=torch.int32).cuda()
    oh, ok, ov = ctx.compact(wl.samples, kept_d, offs_d, offs[-1], dev["hidden"], dev["k"], dev["v"])
    torch.cuda.synchronize()

    class Out:
        out_hidden, out_k, out_v = oh, ok, ov
    for b, s in enumerate(wl.samples):
        check_compaction(wl.steps[0], Out, s, kept[b], offs[b], dtype)
    # a skipped pair stays untouched
    oh2, ok2, ov2 = ctx.compact(wl.samples, kept_d, offs_d, offs[-1], None, dev["k"], None)
    assert oh2 is None and ov2 is None
    torch.cuda.synchronize()
    assert torch.equal(ok2, ok)
    ctx.close()


# ------------------------------------------------------------------ selection on given scores
def test_select_exact_with_ties_and_edge_budgets():
    rng = np.random.default_rng(5)
    cases = [(40, 50, 0.5, 0.5), (1, 300, 1.0, 0.01), (257, 0, 0.3, 0.3), (0, 129, 0.0, 0.7),
             (1000, 1500, 0.1, 0.9), (64, 64, 0.0, 0.0), (33, 95, 1.0, 1.0)]
    for n2, n3, k2r, k3r in cases:
        s = W.layout_2d_3d_txt(0, 7, n2, n3, keep_2d=k2r, keep_3d=k3r)
        ctx = mvla.PruneContext(dtype=torch.float32, n_heads=2, head_dim=64, d_model=64, max_batch=1,
                                max_text=8, max_2d=max(n2, 1), max_3d=max(n3, 1), cold_start_full_keep=0)
        # few distinct values -> many exact ties at the k-th boundary
        attn = rng.integers(1, 6, size=n2 + n3).astype(np.float32)
        attn /= attn.sum()
        out = ctx.select(0, [s], mvla.MODE_FIXED, torch.from_numpy(attn).cuda())
        torch.cuda.synchronize()
        k2, k3 = out.budgets.cpu().numpy()[0]
        assert (k2, k3) == oracle.budget_fixed(s)
        offs = out.out_offsets.cpu().numpy()
        kept = out.kept_idx.cpu().numpy()[:offs[1]]
        ref = oracle.select(oracle.normalise(attn.astype(np.float64), n2, n3), s, int(k2), int(k3))
        assert np.array_equal(kept, ref), (n2, n3)
        assert np.array_equal(out.ahat.cpu().numpy(), attn)
        ctx.close()


def test_select_text_first_and_negative_scores():
    s = W.Sample(seq_off=0, off_txt=0, n_txt=3, off_2d=3, n_2d=200, off_3d=203, n_3d=77,
                 keep_2d=0.25, keep_3d=0.5)
    ctx = mvla.PruneContext(dtype=torch.float32, n_heads=2, head_dim=64, d_model=64, max_batch=1, max_text=8,
                            max_2d=200, max_3d=77, cold_start_full_keep=0)
    rng = np.random.default_rng(1)
    attn = rng.standard_normal(277).astype(np.float32)          # the ordering must hold for any sign
    out = ctx.select(0, [s], mvla.MODE_FIXED, torch.from_numpy(attn).cuda())
    torch.cuda.synchronize()
    kept = out.kept_idx.cpu().numpy()[:out.out_offsets.cpu().numpy()[1]]
    ref = oracle.select(attn.astype(np.float64), s, 50, 39)
    assert np.array_equal(kept, ref)
    ctx.close()


def _scores_of_shape(shape, n, rng):
    """Scores that put the threshold into every part of the selection's histogram: a window around the mean, open ends."""
    if shape == "softmax":                       # what the scoring kernels leave: a bulk below the mean, a few strong ones
        x = np.exp(0.05 * rng.standard_normal(n)) * np.where(rng.random(n) < 0.05, 20.0, 1.0)
        return x / x.sum()
    if shape == "one_token_has_it_all":          # the threshold far below the window
        x = 1e-9 * (1.0 + rng.random(n))
        x[rng.integers(n)] = 1.0
        return x
    if shape == "above_the_window":              # not normalised: everything in the last bin
        return 1e3 + rng.random(n)
    if shape == "narrow":                        # thousands of keys within a few units in the last place, many equal
        return (1.0 + 2.0 ** -23 * rng.integers(0, 40, size=n)) / n
    if shape == "two_scales":                    # one end of the window and the other
        return np.where(rng.random(n) < 0.5, 1e-12, 64.0) * (1.0 + 2.0 ** -20 * rng.integers(0, 1 << 12, size=n))
    x = rng.standard_normal(n) * 10.0 ** rng.integers(-30, 30, size=n).astype(np.float64)       # any float, infinities and zeros
    x[rng.random(n) < 0.1] = 0.0
    x[rng.random(n) < 0.02] = np.inf
    x[rng.random(n) < 0.02] = -np.inf
    return x


@pytest.mark.parametrize("shape", ["softmax", "one_token_has_it_all", "above_the_window", "narrow", "two_scales", "any_float"])
def test_select_finds_the_threshold_wherever_it_lies(shape):
    # sizes around the capacities of the kernel's variants (1024, 2048, 4096 tokens); exact: the k largest, lower index first
    rng = np.random.default_rng(11)
    for n2, n3 in ((1, 1), (0, 2), (31, 33), (512, 512), (513, 512), (1024, 1024), (5, 2044), (1024, 1025), (2048, 2048)):
        ctx = mvla.PruneContext(dtype=torch.float32, n_heads=2, head_dim=64, d_model=64, max_batch=1, max_text=8,
                                max_2d=max(n2, 1), max_3d=max(n3, 1), cold_start_full_keep=0)
        for keep in (0.02, 0.4, 0.97):
            s = W.layout_2d_3d_txt(0, 3, n2, n3, keep_2d=keep, keep_3d=keep)
            attn = _scores_of_shape(shape, n2 + n3, rng).astype(np.float32)
            out = ctx.select(0, [s], mvla.MODE_FIXED, torch.from_numpy(attn).cuda(), flags=mvla.FLAG_RESET_STATE)
            torch.cuda.synchronize()
            k2, k3 = (int(k) for k in out.budgets.cpu().numpy()[0])
            kept = out.kept_idx.cpu().numpy()[:out.out_offsets.cpu().numpy()[1]]
            best2 = np.argsort(-attn[:n2], kind="stable")[:k2]
            best3 = n2 + np.argsort(-attn[n2:], kind="stable")[:k3]
            want = np.concatenate([np.sort(best2), np.sort(best3), n2 + n3 + np.arange(3)])
            assert np.array_equal(kept, want), (shape, n2, n3, keep)
        ctx.close()


@pytest.mark.parametrize("n2,n3", [(400, 500), (700, 1100), (1700, 2300)])
def test_select_with_modalities_that_need_different_numbers_of_histograms(n2, n3):
    # the listed keys of one modality are ranked when the other one's crowded bins are done, too
    rng = np.random.default_rng(12)
    shapes = ["softmax", "one_token_has_it_all", "above_the_window", "narrow", "two_scales", "any_float"]
    ctx = mvla.PruneContext(dtype=torch.float32, n_heads=2, head_dim=64, d_model=64, max_batch=1, max_text=8, max_2d=n2, max_3d=n3,
                            cold_start_full_keep=0)
    for a in shapes:
        for b in shapes + ["equal"]:
            s = W.layout_2d_3d_txt(0, 3, n2, n3, keep_2d=0.35, keep_3d=0.35)
            attn = np.concatenate([_scores_of_shape(a, n2, rng), np.full(n3, 0.5 / n3) if b == "equal" else _scores_of_shape(b, n3, rng)]).astype(np.float32)
            out = ctx.select(0, [s], mvla.MODE_FIXED, torch.from_numpy(attn).cuda(), flags=mvla.FLAG_RESET_STATE)
            torch.cuda.synchronize()
            k2, k3 = (int(k) for k in out.budgets.cpu().numpy()[0])
            kept = out.kept_idx.cpu().numpy()[:out.out_offsets.cpu().numpy()[1]]
            best2 = np.argsort(-attn[:n2], kind="stable")[:k2]
            best3 = n2 + np.argsort(-attn[n2:], kind="stable")[:k3]
            assert np.array_equal(kept, np.concatenate([np.sort(best2), np.sort(best3), n2 + n3 + np.arange(3)])), (a, b)
    ctx.close()


def test_select_takes_no_more_than_one_more_histogram_outside_its_window():
    # Times of 20 selections in a row, in a graph, against scores as the window expects them.  Measured: all equal 1.51, one
    # token with 99 % of the attention 1.64, four fifths zero 1.43; with two or three more histograms 2.99, 2.18 and 3.43.
    # The limit lies between the two.
    n2, n3 = 1536, 2048
    rng = np.random.default_rng(13)
    usual = _scores_of_shape("softmax", n2 + n3, rng)
    sink = 0.01 * usual
    sink[5] += 0.99
    ctx = mvla.PruneContext(dtype=torch.float32, n_heads=2, head_dim=64, d_model=64, max_batch=1, max_text=8, max_2d=n2, max_3d=n3,
                            cold_start_full_keep=0)
    s = W.layout_2d_3d_txt(0, 3, n2, n3, keep_2d=0.4, keep_3d=0.3)
    graphs = []
    for scores in (usual, np.full(n2 + n3, 1.0 / (n2 + n3)), sink, np.where(rng.random(n2 + n3) < 0.8, 0.0, usual)):
        attn = torch.from_numpy(scores.astype(np.float32)).cuda()
        out = ctx.select(0, [s], mvla.MODE_FIXED, attn, flags=mvla.FLAG_RESET_STATE)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(20):
                ctx.select(0, [s], mvla.MODE_FIXED, attn, flags=mvla.FLAG_RESET_STATE, out=out)
        graphs.append((g, attn, out))
    times = [[] for _ in graphs]
    for _ in range(15):
        for (g, _, _), t in zip(graphs, times):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            g.replay()
            a.record()
            g.replay()
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
    usual_ms, *others = [float(np.median(t)) for t in times]
    assert all(t < 1.9 * usual_ms for t in others), (usual_ms, others)
    del graphs
    ctx.close()


# ------------------------------------------------------------------ salience
@pytest.mark.parametrize("dtype,path", [("fp32", mvla.SALIENCE_AUTO), ("bf16", mvla.SALIENCE_FMA),
                                        ("bf16", mvla.SALIENCE_AUTO)])
@pytest.mark.parametrize("text_first", [False, True])
def test_salience_small_ragged(dtype, path, text_first):
    wl = W.small_workload(31, batch=3, D=256, H=4, d=64 if dtype == "fp32" else 128, dtype=dtype,
                          n_txt=(5, 19, 33), n_2d=(70, 130, 1), n_3d=(150, 37, 300), text_first=text_first)
    ctx = mvla.context_for(wl, salience_path=path)
    dev = device_tensors(wl)
    attn, l1 = ctx.salience(wl.samples, dev["q"], dev["k"], dev["hidden"])
    torch.cuda.synchronize()
    attn, l1 = attn.cpu().numpy(), l1.cpu().numpy()
    t = wl.steps[0]
    vis = 0
    for s in wl.samples:
        ref = oracle.salience(t.q, t.k, wl.n_heads, wl.head_dim, s)
        assert_salience_close(attn[vis:vis + s.n_vis], ref)
        assert abs(attn[vis:vis + s.n_vis].sum() - 1.0) < 1e-4
        np.testing.assert_allclose(l1[vis:vis + s.n_vis], oracle.l1norm(t.hidden, wl.d_model, s), rtol=1e-5)
        vis += s.n_vis
    ctx.close()


def test_salience_many_tiles_and_max_text():
    # 2500 keys -> 20 tiles; 64 text queries (the maximum): the streaming kernel in clusters, and the generic one by FMAs with
    # 3 tiles per CTA in a cluster of 7
    wl = W.small_workload(32, batch=1, D=128, H=2, d=128, dtype="bf16", n_txt=(64,), n_2d=(1100,), n_3d=(1400,))
    for path in (mvla.SALIENCE_AUTO, mvla.SALIENCE_FMA):
        ctx = mvla.context_for(wl, salience_path=path)
        dev = device_tensors(wl)
        attn, _ = ctx.salience(wl.samples, dev["q"], dev["k"])
        torch.cuda.synchronize()
        t = wl.steps[0]
        assert_salience_close(attn.cpu().numpy(), oracle.salience(t.q, t.k, 2, 128, wl.samples[0]))
        ctx.close()


def test_tensor_core_and_fma_paths_agree():
    wl = W.config2_single_frame(seed=7)
    dev = device_tensors(wl)
    res = []
    for path in (mvla.SALIENCE_AUTO, mvla.SALIENCE_FMA):
        ctx = mvla.context_for(wl, salience_path=path)
        attn, _ = ctx.salience(wl.samples, dev["q"], dev["k"])
        torch.cuda.synchronize()
        res.append(attn.cpu().numpy())
        ctx.close()
    np.testing.assert_allclose(res[0], res[1], rtol=1e-4, atol=1e-9)


# ------------------------------------------------------------------ the fused step on the five workloads
def _fresh_states(wl):
    return [oracle.State(s.n_vis) for s in wl.samples]


def test_step_config1_tiny_fp32():
    wl = W.config1_tiny()
    ctx = mvla.context_for(wl)
    out, refs = run_and_check_step(ctx, wl, 0, _fresh_states(wl))
    kept = out.kept_idx.cpu().numpy()[:out.total_kept]
    assert np.array_equal(kept, refs[0].kept_idx)
    ctx.close()


@pytest.mark.parametrize("seed", [1, 11, 12, 13])
def test_step_config2_single_frame(seed):
    wl = W.config2_single_frame(seed=seed)
    ctx = mvla.context_for(wl)
    out, refs = run_and_check_step(ctx, wl, 0, _fresh_states(wl))
    assert tuple(out.budgets.cpu().numpy()[0]) == (102, 154)
    assert out.total_kept == 288
    ctx.close()


@pytest.mark.parametrize("seed", [2, 21])
def test_step_config3_multi_view_two_points(seed):
    wl = W.config3_multi_view(seed=seed)
    ctx = mvla.context_for(wl, n_prune_points=2)
    out, refs = run_and_check_step(ctx, wl, 0, _fresh_states(wl), prune_point=0)
    assert out.total_kept == 48 + 448
    # second point: the generator re-projects the rows the ORACLE kept at the first point
    r = refs[0]
    wl2 = W.config3_second_point(wl, r.kept_idx, r.k_2d, r.k_3d)
    out2, refs2 = run_and_check_step(ctx, wl2, 0, _fresh_states(wl2), prune_point=1)
    assert out2.total_kept == 48 + 112
    ctx.close()


def test_step_config4_batched_serving():
    wl = W.config4_batched()
    ctx = mvla.context_for(wl)
    out, refs = run_and_check_step(ctx, wl, 0, _fresh_states(wl))
    offs = out.out_offsets.cpu().numpy()
    assert len(offs) == 17 and (np.diff(offs) > 0).all()
    ctx.close()


def test_step_config5_action_iteration():
    wl = W.config5_action_iteration()
    ctx = mvla.context_for(wl)
    states = _fresh_states(wl)
    s = wl.samples[0]
    for t in range(len(wl.steps)):
        out, refs = run_and_check_step(ctx, wl, t, states, flags=mvla.FLAG_RESET_STATE if t == 0 else 0)
        if t == 0:
            assert out.total_kept == s.seq_len                       # cold start keeps everything
            assert np.array_equal(out.kept_idx.cpu().numpy()[:s.seq_len], np.arange(s.seq_len))
        else:
            assert out.total_kept == s.n_txt + 384
        assert diag_records(out, 1)[0]["t"] == t + 1
    ctx.close()


def test_step_small_ragged_batch_with_state_and_dry_run():
    wl = W.small_workload(41, batch=3, D=256, H=4, d=128, dtype="bf16", n_txt=(5, 19, 33),
                          n_2d=(70, 130, 260), n_3d=(150, 37, 300), keep=(0.4, 0.3, 0.55), steps=9,
                          cold_start=1)
    ctx = mvla.context_for(wl)
    states = _fresh_states(wl)
    for t in range(9):                                                # crosses the Eq. 8 -> Eq. 9 switch at t = 7
        out, refs = run_and_check_step(ctx, wl, t, states)
        if t == 3:                                                    # a dry run leaves state and t untouched
            dev = device_tensors(wl, t)
            dry = ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"],
                                 flags=mvla.FLAG_NO_STATE_UPDATE)
            torch.cuda.synchronize()
            assert diag_records(dry, 3)[0]["t"] == 5
    ctx.close()


@pytest.mark.parametrize("scale,expect", [(0.05, mvla.SET_2D), (0.136, mvla.SET_2D | mvla.SET_3D), (0.30, mvla.SET_3D)])
def test_paper_default_thresholds_all_three_branches(scale, expect):
    # 3D hidden rows scaled by s give a feature-norm share of about s/(1+s): 0.048, 0.12, 0.23 against
    # the paper's default thresholds 0.08 / 0.20
    wl = W.small_workload(51, batch=1, D=512, H=4, d=128, dtype="bf16", n_txt=(9,), n_2d=(200,), n_3d=(280,),
                          keep=(0.35,), scale_3d=scale, spike_frac=0.0)
    wl.tau_2d, wl.tau_3d = 0.08, 0.20
    ctx = mvla.context_for(wl)
    out, refs = run_and_check_step(ctx, wl, 0, _fresh_states(wl))
    assert diag_records(out, 1)[0]["c_s1"] == expect == refs[0].c_s1
    ctx.close()


def test_results_are_deterministic():
    wl = W.config2_single_frame(seed=3)
    ctx = mvla.context_for(wl)
    dev = device_tensors(wl)
    outs = []
    for _ in range(3):
        o = ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"],
                           flags=mvla.FLAG_RESET_STATE)
        torch.cuda.synchronize()
        n = o.total_kept                                            # rows past it are unwritten scratch
        outs.append((o.attn.clone(), o.kept_idx[:n].clone(), o.out_hidden[:n].clone(), o.out_k[:n].clone()))
    for a in outs[1:]:
        assert all(torch.equal(x, y) for x, y in zip(a, outs[0]))
    ctx.close()


# ------------------------------------------------------------------ boundary behaviour
def test_error_codes_never_fault():
    wl = W.small_workload(61, batch=2, D=256, H=4, d=128, dtype="bf16")
    ctx = mvla.context_for(wl)
    dev = device_tensors(wl)
    good = list(wl.samples)

    def code(fn):
        with pytest.raises(mvla.MvlaError) as e:
            fn()
        return e.value.code

    import copy
    bad = copy.deepcopy(good); bad[0].n_txt = 0
    assert code(lambda: ctx.salience(bad, dev["q"], dev["k"])) == mvla.ERR_INVALID_ARG
    bad = copy.deepcopy(good); bad[0].off_3d = bad[0].off_2d          # overlapping segments
    assert code(lambda: ctx.salience(bad, dev["q"], dev["k"])) == mvla.ERR_INVALID_ARG
    bad = copy.deepcopy(good); bad[1].n_2d = 10 ** 6
    assert code(lambda: ctx.salience(bad, dev["q"], dev["k"])) == mvla.ERR_CAPACITY
    bad = copy.deepcopy(good); bad[1].seq_off = 10 ** 6               # beyond the rows given
    assert code(lambda: ctx.salience(bad, dev["q"], dev["k"])) == mvla.ERR_INVALID_ARG
    bad = copy.deepcopy(good); bad[1].state_slot = bad[0].state_slot  # two writers of one state
    assert code(lambda: ctx.prune_step(0, bad, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])) == mvla.ERR_STATE
    assert code(lambda: ctx.prune_step(3, good, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])) == mvla.ERR_STATE
    assert code(lambda: ctx.prune_step(0, good, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"], flags=8)) == mvla.ERR_INVALID_ARG
    assert code(lambda: ctx.prune_step(0, good * 2, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])) == mvla.ERR_CAPACITY
    misaligned = dev["q"].view(-1)[1:1 + dev["q"].numel() - 8].contiguous()
    # .contiguous() of a slice is a fresh allocation, so build a truly misaligned pointer by hand
    import ctypes as C
    cs = mvla.c_samples(good)
    rc = ctx._lib.mvla_salience(ctx._h, 2, cs, dev["q"].data_ptr() + 2, dev["k"].data_ptr(), None,
                                dev["q"].shape[0], torch.empty(1000, device="cuda").data_ptr(), None, 0)
    assert rc == mvla.ERR_INVALID_ARG
    # the context is still usable afterwards
    ctx.prune_step(0, good, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])
    torch.cuda.synchronize()
    ctx.close()
    with pytest.raises(mvla.MvlaError) as e:
        mvla.PruneContext(dtype=torch.bfloat16, n_heads=4, head_dim=48, d_model=256, max_batch=1, max_text=8,
                          max_2d=8, max_3d=8)
    assert e.value.code == mvla.ERR_UNSUPPORTED


def test_inputs_stable_flag_changes_timing_only():
    # back-to-back steps on rotating buffers, with and without the promise that the inputs are not
    # produced by the preceding work: identical results, step after step
    wls = [W.config2_single_frame(seed=s) for s in (31, 32, 33)]
    wl = wls[0]
    ctx = mvla.context_for(wl)
    devs = [device_tensors(w) for w in wls]
    ref = []
    for d in devs:
        o = ctx.prune_step(0, wl.samples, wl.mode, d["q"], d["k"], d["v"], d["hidden"], flags=mvla.FLAG_RESET_STATE)
        torch.cuda.synchronize()
        n = o.total_kept
        ref.append((o.attn.clone(), o.kept_idx[:n].clone(), o.out_hidden[:n].clone(), o.out_v[:n].clone()))
    outs = [ctx.alloc_outputs(wl.samples, extras=True) for _ in range(3)]
    for rep in range(30):                                   # no synchronisation between the steps
        i = rep % 3
        d = devs[i]
        ctx.prune_step(0, wl.samples, wl.mode, d["q"], d["k"], d["v"], d["hidden"],
                       flags=mvla.FLAG_RESET_STATE | mvla.FLAG_INPUTS_STABLE, out=outs[i])
    torch.cuda.synchronize()
    for i in range(3):
        o, n = outs[i], len(ref[i][1])
        got = (o.attn, o.kept_idx[:n], o.out_hidden[:n], o.out_v[:n])
        assert all(torch.equal(x, y) for x, y in zip(got, ref[i]))
    ctx.close()


def test_pipelined_steps_with_state_match_serial_steps():
    # action steps with carry-over, enqueued back to back without synchronisation and with the
    # stable-inputs promise (scoring, selection and row copy of neighbouring steps overlap), against the
    # same steps run one at a time: identical bits, including when output buffers are reused
    wl = W.small_workload(43, batch=3, D=256, H=4, d=128, dtype="bf16", n_txt=(5, 19, 33), n_2d=(70, 130, 260),
                          n_3d=(150, 37, 300), keep=(0.4, 0.3, 0.55), steps=10, cold_start=1)
    devs = [device_tensors(wl, t) for t in range(10)]

    def run(flag, n_out, sync):
        ctx = mvla.context_for(wl)
        outs = [ctx.alloc_outputs(wl.samples, extras=True) for _ in range(n_out)]
        res = []
        for t, d in enumerate(devs):
            o = ctx.prune_step(0, wl.samples, wl.mode, d["q"], d["k"], d["v"], d["hidden"],
                               flags=flag | (mvla.FLAG_RESET_STATE if t == 0 else 0), out=outs[t % n_out])
            if sync:
                torch.cuda.synchronize()
            res.append((o.total_kept, t % n_out))
        torch.cuda.synchronize()
        snap = [None] * 10
        for t in range(10 - n_out, 10):                       # the last n_out steps are still in their buffers
            o, n = outs[t % n_out], res[t][0]
            snap[t] = (o.ahat.clone(), o.kept_idx[:n].clone(), o.budgets.clone(), o.out_hidden[:n].clone(),
                       o.out_k[:n].clone())
        ctx.close()
        return snap

    ref = run(0, 10, True)
    for n_out in (10, 3, 2, 1):                                # 1: every step reuses the same output buffers
        got = run(mvla.FLAG_INPUTS_STABLE, n_out, False)
        for t in range(10 - n_out, 10):
            assert all(torch.equal(x, y) for x, y in zip(got[t], ref[t])), (n_out, t)


def test_pipelined_steps_sharing_an_index_buffer_two_steps_apart():
    # Every step has its own row buffers, but steps t and t + 2 share kept_idx, and the caller's stream is
    # kept busy between the steps so that the row copies lag behind the selections running ahead on the
    # library's own streams.  A selection must not overwrite indices that an earlier copy has yet to read.
    import dataclasses
    wl = W.small_workload(47, batch=2, D=256, H=4, d=128, dtype="bf16", n_txt=(7, 21), n_2d=(90, 200),
                          n_3d=(160, 310), keep=(0.45, 0.35), steps=12, cold_start=0)
    devs = [device_tensors(wl, t) for t in range(12)]

    def run(flag, share, delay):
        ctx = mvla.context_for(wl)
        outs = [ctx.alloc_outputs(wl.samples, extras=True) for _ in range(12)]
        if share:
            outs = [dataclasses.replace(o, kept_idx=outs[t % 2].kept_idx) for t, o in enumerate(outs)]
        kept = []
        for t, d in enumerate(devs):
            if delay:
                torch.cuda._sleep(300000)                     # touches none of the step's buffers
            o = ctx.prune_step(0, wl.samples, wl.mode, d["q"], d["k"], d["v"], d["hidden"],
                               flags=flag | (mvla.FLAG_RESET_STATE if t == 0 else 0), out=outs[t])
            kept.append(o.total_kept)
            if not flag:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        res = [(o.out_hidden[:n].clone(), o.out_k[:n].clone(), o.budgets.clone()) for o, n in zip(outs, kept)]
        ctx.close()
        return res

    ref = run(0, False, False)
    got = run(mvla.FLAG_INPUTS_STABLE, True, True)
    for t in range(12):
        assert all(torch.equal(x, y) for x, y in zip(got[t], ref[t])), t


def test_pipelined_steps_of_interleaved_episodes_keep_their_states_apart():
    # three episodes (state slots) take turns; inside an episode the carry-over must see the steps in
    # call order although selections of different episodes are free to run beside one another
    import dataclasses
    wl = W.small_workload(53, batch=2, D=256, H=4, d=128, dtype="bf16", n_txt=(9, 30), n_2d=(100, 180),
                          n_3d=(140, 333), keep=(0.5, 0.3), steps=12, cold_start=1)
    devs = [device_tensors(wl, t) for t in range(12)]
    episodes = [[dataclasses.replace(s, state_slot=s.state_slot + 2 * e) for s in wl.samples] for e in range(3)]
    order = [0, 1, 2, 0, 0, 1, 2, 2, 1, 0, 2, 1]              # which episode each call belongs to

    def run(flag):
        ctx = mvla.context_for(wl, n_state_slots=6)
        outs = [ctx.alloc_outputs(wl.samples, extras=True) for _ in range(12)]
        seen, kept = set(), []
        for t, e in enumerate(order):
            d = devs[t]
            o = ctx.prune_step(0, episodes[e], wl.mode, d["q"], d["k"], d["v"], d["hidden"],
                               flags=flag | (0 if e in seen else mvla.FLAG_RESET_STATE), out=outs[t])
            seen.add(e)
            kept.append(o.total_kept)
            if not flag:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        res = [(o.ahat.clone(), o.kept_idx[:n].clone(), o.budgets.clone(), o.out_v[:n].clone())
               for o, n in zip(outs, kept)]
        ctx.close()
        return res

    ref, got = run(0), run(mvla.FLAG_INPUTS_STABLE)
    for t in range(12):
        assert all(torch.equal(x, y) for x, y in zip(got[t], ref[t])), t


@pytest.mark.parametrize("text_first", [False, True])
def test_chained_requests_match_serial_steps(text_first):
    # Requests of one sample with stable inputs are chained: the scores of a step are taken beside the selection and row copy of
    # the step before.  A sequence that mixes independent episodes, carried-over state, fixed and adaptive budgets, steps without
    # row copy, steps whose inputs are an earlier step's output rows, and a step without the promise: the same bits as one at a time.
    wl = W.small_workload(59, batch=1, D=512, H=4, d=128, dtype="bf16", n_txt=(21,), n_2d=(200,), n_3d=(333,), keep=(0.4,), steps=16,
                          text_first=text_first)
    devs = [device_tensors(wl, t) for t in range(16)]
    s = wl.samples[0]
    import dataclasses

    def run(flag, sync):
        ctx = mvla.context_for(wl, n_state_slots=3)
        outs, kept = [], []
        for t in range(16):
            d, sample = devs[t], dataclasses.replace(s, state_slot=t % 3)
            mode = mvla.MODE_FIXED if t % 4 == 1 else mvla.MODE_ADAPTIVE
            rows = t % 5 != 3
            if t in (6, 7, 12):                                # the rows that an earlier step kept, pruned again
                prev, n = outs[t - 1 - t % 2], kept[t - 1 - t % 2]
                q, k, v, h = d["q"][:n], prev.out_k[:n], prev.out_v[:n], prev.out_hidden[:n]
                n3 = (n - s.n_txt) // 2
                sample = W.layout_2d_3d_txt(0, s.n_txt, n - s.n_txt - n3, n3, keep_2d=0.5, keep_3d=0.3, keep_total=0.4, state_slot=t % 3)
            else:
                q, k, v, h = (d[x] for x in ("q", "k", "v", "hidden"))
            o = ctx.alloc_outputs([sample], hidden=rows, kv=rows, extras=True)
            ctx.prune_step(0, [sample], mode, q, k, v if rows else None, h,
                           flags=(0 if t == 9 else flag) | (mvla.FLAG_RESET_STATE if t < 3 or t in (6, 7, 12) else 0), out=o)
            outs.append(o)
            kept.append(o.total_kept)
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        ctx.close()
        return [(o.ahat, o.kept_idx[:n], o.budgets, o.out_offsets) + ((o.out_hidden[:n], o.out_k[:n], o.out_v[:n]) if o.out_hidden is not None else ())
                for o, n in zip(outs, kept)]

    ref = run(0, True)
    for _ in range(3):
        got = run(mvla.FLAG_INPUTS_STABLE, False)
        for t in range(16):
            assert len(got[t]) == len(ref[t]) and all(torch.equal(x, y) for x, y in zip(got[t], ref[t])), t


@pytest.mark.parametrize("mode", [mvla.MODE_FIXED, mvla.MODE_ADAPTIVE])
@pytest.mark.parametrize("shape", [
    dict(H=4, d=128, n_txt=(5,)),                                   # 16, 32 and 64 tensor-memory columns
    dict(H=4, d=128, n_txt=(32,)),
    dict(H=4, d=128, n_txt=(64,)),
    dict(H=8, d=64, n_txt=(33,), n_kv_heads=2),
    dict(H=4, d=96, n_txt=(17,), dtype="fp8"),
    dict(H=64, d=64, n_txt=(21,), n_2d=(500,), n_3d=(400,)),        # 512 scoring CTAs: the streaming kernel, in a chained step
], ids=lambda s: f"{s['H']}x{s['d']}_text{s['n_txt'][0]}_{s.get('dtype', 'bf16')}_kv{s.get('n_kv_heads', 0)}")
def test_chained_steps_of_one_episode_match_serial_steps(shape, mode):
    # every step carries over the state of the step directly before it, whose tail its scores are taken beside
    wl = W.small_workload(67, **{**dict(batch=1, D=256, dtype="bf16", n_2d=(129,), n_3d=(383,), keep=(0.2,), keep_fixed=(0.25, 0.15),
                                        steps=14, cold_start=1), **shape})
    devs = [device_tensors(wl, t) for t in range(14)]

    def run(flag):
        ctx = mvla.context_for(wl)
        outs = [ctx.alloc_outputs(wl.samples, extras=True) for _ in range(14)]
        torch.cuda.synchronize()
        if flag:
            torch.cuda._sleep(2_000_000)          # the host runs ahead: the steps follow one another on the GPU
        for t, (d, o) in enumerate(zip(devs, outs)):
            ctx.prune_step(0, wl.samples, mode, d["q"], d["k"], d["v"], d["hidden"], flags=flag | (mvla.FLAG_RESET_STATE if t == 0 else 0), out=o)
            if not flag:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        ctx.close()
        as_bytes = lambda x: x.contiguous().view(torch.uint8)
        return [(o.attn, o.ahat, o.z, o.budgets, o.diag, o.kept_idx[:o.total_kept]) +
                tuple(as_bytes(x[:o.total_kept]) for x in (o.out_hidden, o.out_k, o.out_v)) for o in outs]

    ref, got = run(0), run(mvla.FLAG_INPUTS_STABLE)
    for t in range(14):
        assert all(torch.equal(x, y) for x, y in zip(got[t], ref[t])), t


@pytest.mark.parametrize("seed", range(4))
def test_chained_forked_and_unpromised_calls_in_one_context_match_serial_calls(seed):
    # One sample (chained on the caller's stream), two samples (forked to the side streams), steps without the promise, dry
    # runs and mvla_select in an order drawn at random, on shared state slots, through every scratch set several times, with
    # inputs that one of the last eight calls has written and output buffers used again: the same bits as one at a time.
    import dataclasses
    wl = W.small_workload(71, batch=2, D=256, H=4, d=128, dtype="bf16", n_txt=(21, 9), n_2d=(130,), n_3d=(190,), keep=(0.4, 0.3), steps=6)
    devs = [device_tensors(wl, t) for t in range(6)]
    n_calls, n_out = 64, 16
    rng = np.random.default_rng(seed)
    calls = []
    for t in range(n_calls):
        kind = ("chain", "fork", "plain", "dry", "select")[rng.choice(5, p=[0.4, 0.35, 0.1, 0.08, 0.07])]
        slots = [int(x) for x in rng.permutation(4)[:1 if kind in ("chain", "select") else 2]]
        back = t - int(rng.integers(1, 9))
        source = back if back >= 0 and kind != "select" and calls[back][0] != "select" and rng.random() < 0.4 else -1
        if source < 0:
            samples = [dataclasses.replace(wl.samples[i], state_slot=slot) for i, slot in enumerate(slots)]
        else:                                                 # in the first 100 rows of an earlier call's outputs, states of their own
            samples = [W.layout_2d_3d_txt(50 * i, 10, 15, 25, keep_2d=0.5, keep_3d=0.3, keep_total=0.4, state_slot=4 + slot)
                       for i, slot in enumerate(slots)]
        calls.append((kind, samples, source, mvla.MODE_FIXED if rng.random() < 0.5 else mvla.MODE_ADAPTIVE, rng.random() < 0.3))
    scores = torch.from_numpy(rng.random(320).astype(np.float32)).cuda()

    def run(flag):
        ctx = mvla.context_for(wl, n_state_slots=8)
        bufs = [ctx.alloc_outputs(wl.samples, extras=True) for _ in range(n_out)]
        for o in bufs:
            for x in (o.out_hidden, o.out_k, o.out_v):
                x.zero_()
        torch.cuda.synchronize()
        for t, (kind, samples, source, mode, busy) in enumerate(calls):
            d, o = devs[t % 6], bufs[t % n_out]
            if flag and busy:
                torch.cuda._sleep(200_000)                    # touches none of the calls' buffers
            if kind == "select":
                ctx.select(0, samples, mvla.MODE_FIXED, scores, out=o)
                o.total_kept = 0                              # (no rows)
            else:
                p = bufs[source % n_out]
                q, k, v, h = ((d["q"], d["k"], d["v"], d["hidden"]) if source < 0 else
                              (d["q"][:100], p.out_k[:100], p.out_v[:100], p.out_hidden[:100]))
                ctx.prune_step(0, samples, mode, q, k, v, h, out=o,
                               flags=mvla.FLAG_NO_STATE_UPDATE if kind == "dry" else flag if kind in ("chain", "fork") else 0)
            if not flag:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        ctx.close()
        return bufs

    ref, got = run(0), run(mvla.FLAG_INPUTS_STABLE)
    for t in range(n_calls - n_out, n_calls):
        kind, samples = calls[t][:2]
        a, b = ref[t % n_out], got[t % n_out]
        n_vis, n, m = sum(s.n_2d + s.n_3d for s in samples), len(samples), a.total_kept
        listed = int(a.out_offsets[n])
        for x, y in ((a.ahat[:n_vis], b.ahat[:n_vis]), (a.out_offsets[:n + 1], b.out_offsets[:n + 1]), (a.budgets[:n], b.budgets[:n]),
                     (a.kept_idx[:listed], b.kept_idx[:listed]), (a.out_hidden[:m], b.out_hidden[:m]), (a.out_k[:m], b.out_k[:m]),
                     (a.out_v[:m], b.out_v[:m])):
            assert torch.equal(x, y), (t, kind)


@pytest.mark.parametrize("reads", ["state", "rows"])
def test_stable_steps_are_ordered_after_a_call_without_the_promise(reads):
    # Six stable batches, so that every scratch set has events of its own; a call without the promise, kept from running for 10 ms; a
    # stable step that has nothing to do with it; then a stable batch that reads what that call writes: the smoothed
    # states of its slots, or the rows that it kept.  Each of six more batches runs on another scratch set.
    import dataclasses
    wl = W.small_workload(61, batch=2, D=256, H=4, d=128, dtype="bf16", n_txt=(9, 30), n_2d=(100, 180), n_3d=(140, 333),
                          keep=(0.5, 0.3), steps=14, cold_start=0)
    devs = [device_tensors(wl, t) for t in range(14)]

    def slots(first):
        return [dataclasses.replace(s, state_slot=first + i) for i, s in enumerate(wl.samples)]

    def run(flag):
        ctx = mvla.context_for(wl, n_state_slots=6)
        outs, kept, late = [], [], None
        for t in range(14):
            q, k, v, h = (devs[t][x] for x in ("q", "k", "v", "hidden"))
            samples = slots(4 if t < 6 else 0)
            if t == 7:
                samples = slots(2)[:1]                        # one sample: chained on the caller's stream
            if reads == "rows" and t > 7:                     # the rows that call 6 kept, pruned again
                k, v, h = late.out_k, late.out_v, late.out_hidden
            o = ctx.alloc_outputs(samples, extras=True)
            if t == 6:
                late = o
                for x in (o.out_k, o.out_v, o.out_hidden):
                    x.zero_()
                torch.cuda.synchronize()
                if flag:
                    torch.cuda._sleep(20_000_000)
            ctx.prune_step(0, samples, wl.mode, q, k, v, h, flags=(0 if t == 6 else flag) | (mvla.FLAG_RESET_STATE if t in (0, 7) else 0), out=o)
            outs.append(o)
            kept.append(o.total_kept)
            if not flag:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        ctx.close()
        return [(o.ahat, o.kept_idx[:n], o.budgets, o.out_hidden[:n], o.out_v[:n]) for o, n in zip(outs, kept)]

    ref, got = run(0), run(mvla.FLAG_INPUTS_STABLE)
    for t in range(14):
        assert all(torch.equal(x, y) for x, y in zip(got[t], ref[t])), t


def test_step_segments_in_order_3d_text_2d():
    # the three segments may come in any order; here [3D | text | 2D], two samples, adaptive budgets
    base = W.small_workload(47, batch=2, D=256, H=4, d=128, dtype="bf16", n_txt=(9, 30), n_2d=(140, 77),
                            n_3d=(200, 301), keep=(0.4, 0.3))
    t = base.steps[0]
    order, samples = [], []
    for s in base.samples:
        r = s.seq_off
        order += list(range(r + s.off_3d, r + s.off_3d + s.n_3d)) + list(range(r + s.off_txt, r + s.off_txt + s.n_txt)) \
            + list(range(r + s.off_2d, r + s.off_2d + s.n_2d))
        samples.append(W.Sample(seq_off=s.seq_off, off_3d=0, n_3d=s.n_3d, off_txt=s.n_3d, n_txt=s.n_txt,
                                off_2d=s.n_3d + s.n_txt, n_2d=s.n_2d, keep_total=s.keep_total,
                                state_slot=s.state_slot))
    order = np.array(order)
    ten = W.Tensors(hidden=np.ascontiguousarray(t.hidden[order]), q=np.ascontiguousarray(t.q[order]),
                    k=np.ascontiguousarray(t.k[order]), v=np.ascontiguousarray(t.v[order]))
    wl = W.Workload("segments_3d_txt_2d", base.dtype, base.n_heads, base.head_dim, base.d_model, base.mode,
                    samples, [ten])
    ctx = mvla.context_for(wl)
    out, refs = run_and_check_step(ctx, wl, 0, _fresh_states(wl))
    ctx.close()


@pytest.mark.parametrize("dtype,path", [("bf16", mvla.SALIENCE_AUTO), ("bf16", mvla.SALIENCE_FMA), ("fp32", mvla.SALIENCE_AUTO)])
def test_grouped_key_heads(dtype, path):
    # 8 query heads read 2 key heads: K and V rows are a quarter as wide as Q rows
    wl = W.small_workload(17, batch=2, D=256, H=8, d=64, dtype=dtype, mode=W.MODE_FIXED, n_txt=(9, 33),
                          n_2d=(130, 70), n_3d=(150, 300), n_kv_heads=2)
    t = wl.steps[0]
    assert t.k.shape[1] == 2 and t.q.shape[1] == 8
    ctx = mvla.context_for(wl, salience_path=path)
    dev = device_tensors(wl)
    attn, _ = ctx.salience(wl.samples, dev["q"], dev["k"])
    out = ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])
    torch.cuda.synchronize()
    attn, attn_step = attn.cpu().numpy(), out.attn.cpu().numpy()
    offs, kept_all, budgets = out.out_offsets.cpu().numpy(), out.kept_idx.cpu().numpy(), out.budgets.cpu().numpy()
    vis = 0
    for b, s in enumerate(wl.samples):
        ref = oracle.salience_gqa(t.q, t.k, 8, 2, 64, s)
        assert_salience_close(attn[vis:vis + s.n_vis], ref, "stand-alone scores")
        assert_salience_close(attn_step[vis:vis + s.n_vis], ref, "scores of the fused step")
        k2, k3 = oracle.budget_fixed(s)
        assert (int(budgets[b, 0]), int(budgets[b, 1])) == (k2, k3)
        kept = kept_all[offs[b]:offs[b + 1]]
        check_kept_against_oracle(s, kept, k2, k3, oracle.normalise(ref, s.n_2d, s.n_3d))
        check_stagewise_exact(s, kept, k2, k3, out.ahat.cpu().numpy()[vis:vis + s.n_vis])
        check_compaction(t, out, s, kept, int(offs[b]), wl.dtype)        # K / V rows of 2 x 64 elements
        vis += s.n_vis
    ctx.close()


@pytest.mark.parametrize("d", [96, 160, 256])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_other_head_dims(dtype, d):
    # 96 and 160 are not multiples of the 64-element TMA box: the last box is partly out of range and zero-filled
    wl = W.small_workload(19, batch=2, D=512, H=2, d=d, dtype=dtype, n_txt=(7, 30), n_2d=(140, 60), n_3d=(100, 270))
    ctx = mvla.context_for(wl)
    run_and_check_step(ctx, wl, 0, [oracle.State(s.n_vis) for s in wl.samples])
    ctx.close()


@pytest.mark.parametrize("mode", [W.MODE_FIXED, W.MODE_ADAPTIVE])
def test_step_with_an_empty_modality(mode):
    # one sample without 2D tokens, one without 3D tokens, one ordinary
    wl = W.small_workload(23, batch=3, D=256, H=4, d=64, dtype="bf16", mode=mode, n_txt=(6, 17, 9),
                          n_2d=(0, 150, 40), n_3d=(200, 0, 70))
    ctx = mvla.context_for(wl)
    out, refs = run_and_check_step(ctx, wl, 0, [oracle.State(s.n_vis) for s in wl.samples])
    b = out.budgets.cpu().numpy()
    assert b[0, 0] == 0 and b[1, 1] == 0
    ctx.close()


def test_step_more_samples_than_one_launch_carries():
    # 40 samples: the per-sample descriptors travel 32 to a launch, so every stage runs in two launches
    wl = W.small_workload(29, batch=40, D=128, H=2, d=64, dtype="bf16", n_txt=(3, 11, 6), n_2d=(33, 140, 64),
                          n_3d=(129, 20, 75), keep=(0.3, 0.5, 0.25))
    ctx = mvla.context_for(wl)
    states = [oracle.State(s.n_vis) for s in wl.samples]
    run_and_check_step(ctx, wl, 0, states)
    ctx.close()


def test_step_at_the_capacity_limits():
    # 64 text tokens, 2048 + 2048 visual tokens: 32 key tiles, four per CTA in a cluster of eight
    wl = W.small_workload(37, batch=1, D=64, H=1, d=64, dtype="bf16", n_txt=(64,), n_2d=(2048,), n_3d=(2048,),
                          keep=(0.1,))
    ctx = mvla.context_for(wl)
    run_and_check_step(ctx, wl, 0, [oracle.State(s.n_vis) for s in wl.samples])
    ctx.close()


def test_head_sharded_step_two_ranks_emulated_on_one_gpu():
    # Tensor-parallel serving: each rank scores its own heads, the scores are averaged over the ranks, every
    # rank selects on the same scores and copies its own K / V heads.  The two ranks run one after the other
    # here (their kernels do not wait on one another); the average is taken in place of the all-reduce.
    from paper_2604_09244_b200 import tensor_parallel as TP
    wl = W.small_workload(73, batch=2, D=256, H=8, d=64, dtype="bf16", mode=W.MODE_FIXED, n_txt=(9, 20),
                          n_2d=(130, 64), n_3d=(200, 300), n_kv_heads=4)
    t = wl.steps[0]
    dev = device_tensors(wl)
    world = 2
    ctxs, shards, partial = [], [], []
    for r in range(world):
        ctx = mvla.PruneContext(dtype=torch.bfloat16, n_heads=8 // world, n_kv_heads=4 // world, head_dim=64, d_model=256,
                                max_batch=2, max_text=32, max_2d=256, max_3d=512, tau_2d=wl.tau_2d, tau_3d=wl.tau_3d,
                                cold_start_full_keep=0)
        sh = {n: TP.head_shard(dev[n], r, world) for n in ("q", "k", "v")}
        a, _ = ctx.salience(wl.samples, sh["q"], sh["k"])
        ctxs.append(ctx); shards.append(sh); partial.append(a)
    torch.cuda.synchronize()
    attn = (partial[0] + partial[1]) / world                    # what the all-reduce leaves on every rank
    vis = 0
    for s in wl.samples:
        assert_salience_close(attn[vis:vis + s.n_vis].cpu().numpy(), oracle.salience_gqa(t.q, t.k, 8, 4, 64, s))
        vis += s.n_vis
    kept_by_rank = []
    for r in range(world):
        out = ctxs[r].alloc_outputs(wl.samples, extras=True)
        ctxs[r].select(0, wl.samples, wl.mode, attn, None, out=out)
        total = sum(s.seq_len for s in wl.samples)
        ctxs[r].compact(wl.samples, out.kept_idx, out.out_offsets, total, dev["hidden"], shards[r]["k"], shards[r]["v"],
                        out_hidden=out.out_hidden, out_k=out.out_k, out_v=out.out_v)
        torch.cuda.synchronize()
        offs, kept_all = out.out_offsets.cpu().numpy(), out.kept_idx.cpu().numpy()
        kept_by_rank.append(kept_all[:offs[-1]].copy())
        vis = 0
        for b, s in enumerate(wl.samples):
            kept = kept_all[offs[b]:offs[b + 1]]
            k2, k3 = oracle.budget_fixed(s)
            check_kept_against_oracle(s, kept, k2, k3, oracle.normalise(oracle.salience_gqa(t.q, t.k, 8, 4, 64, s), s.n_2d, s.n_3d))
            n = len(kept)
            rows = s.seq_off + kept
            assert torch.equal(out.out_hidden[offs[b]:offs[b] + n], dev["hidden"][rows])
            assert torch.equal(out.out_k[offs[b]:offs[b] + n], shards[r]["k"][rows])       # this rank's key heads
            assert torch.equal(out.out_v[offs[b]:offs[b] + n], shards[r]["v"][rows])
            vis += s.n_vis
    assert np.array_equal(kept_by_rank[0], kept_by_rank[1])      # identical scores, identical decisions
    # the packaged call on a group of one rank: same kept positions as the ranks above
    full = mvla.context_for(wl)
    o = TP.prune_step_head_sharded(full, 0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])
    torch.cuda.synchronize()
    n = int(o.out_offsets[-1])
    assert np.array_equal(o.kept_idx[:n].cpu().numpy(), kept_by_rank[0])
    for c in ctxs + [full]:
        c.close()


def test_fp8_keys_small_ragged_and_grouped():
    # q, k, v in e4m3 (hidden bf16): ragged tiles, two samples, grouped key heads, head_dim 64 and 128
    for d, hkv in ((128, 0), (64, 2)):
        wl = W.small_workload(81, batch=2, D=256, H=4, d=d, dtype="fp8", n_txt=(7, 33), n_2d=(130, 70), n_3d=(150, 300),
                              n_kv_heads=hkv)
        ctx = mvla.context_for(wl)
        dev = device_tensors(wl)
        assert dev["k"].dtype == torch.float8_e4m3fn and dev["hidden"].dtype == torch.bfloat16
        attn, l1 = ctx.salience(wl.samples, dev["q"], dev["k"], dev["hidden"])
        torch.cuda.synchronize()
        attn = attn.cpu().numpy()
        t = wl.steps[0]
        vis = 0
        for s in wl.samples:
            ref = oracle.salience_gqa(t.q, t.k, 4, hkv or 4, d, s)
            assert_salience_close(attn[vis:vis + s.n_vis], ref, "e4m3 scores")
            vis += s.n_vis
        if not hkv:
            run_and_check_step(ctx, wl, 0, [oracle.State(s.n_vis) for s in wl.samples])
        ctx.close()


def test_fp8_step_single_frame_shape():
    wl = W.config2_single_frame(dtype="fp8")          # 32 text + 256 2D + 512 3D, D = 4096, 32 heads x 128
    ctx = mvla.context_for(wl)
    run_and_check_step(ctx, wl, 0, [oracle.State(s.n_vis) for s in wl.samples])
    ctx.close()


# ------------------------------------------------------------------ fused tail: ties, guard bands, bounded waits
def _duplicate_visual_rows(wl, group):
    """Make groups of `group` neighbouring visual tokens identical (hidden, q, k, v): tokens of one 128-key
    tile then get bit-identical scores, so the selection has to fall back on the index."""
    t = wl.steps[0]
    for s in wl.samples:
        for off, n in ((s.off_2d, s.n_2d), (s.off_3d, s.n_3d)):
            rows = s.seq_off + off + np.arange(n)
            src = s.seq_off + off + (np.arange(n) // group) * group
            for name in ("hidden", "q", "k", "v"):
                getattr(t, name)[rows] = getattr(t, name)[src]


@pytest.mark.parametrize("mode", [W.MODE_FIXED, W.MODE_ADAPTIVE])
@pytest.mark.parametrize("sizes", [((200, 77), (300, 500)), ((900, 1000), (1100, 130))])   # <= 1024 and <= 2048 tokens
@pytest.mark.parametrize("group", [8, 4096])                                                  # runs of 8; everything equal
def test_step_with_equal_scores_straddling_the_budget(mode, sizes, group):
    wl = W.small_workload(91, batch=2, D=256, H=2, d=64, dtype="bf16", mode=mode, n_txt=(9, 20), n_2d=sizes[0],
                          n_3d=sizes[1], keep=(0.37, 0.21), keep_fixed=(0.33, 0.41))
    _duplicate_visual_rows(wl, group)
    ctx = mvla.context_for(wl)
    out, refs = run_and_check_step(ctx, wl, 0, _fresh_states(wl))     # includes the exact stage-wise check
    ahat = out.ahat.cpu().numpy()
    assert len(np.unique(ahat)) < 0.6 * len(ahat), "the case was meant to hold many equal scores"
    ctx.close()


def test_step_leaves_the_bytes_behind_its_outputs_alone():
    # stands in for a memory checker: capacity-sized output buffers are filled with a pattern, and whatever
    # lies behind the rows / list entries the step reports must still hold it afterwards
    wl = W.small_workload(93, batch=3, D=256, H=4, d=128, dtype="bf16", n_txt=(5, 19, 33), n_2d=(70, 130, 260),
                          n_3d=(150, 37, 300), keep=(0.4, 0.3, 0.55))
    ctx = mvla.context_for(wl)
    dev = device_tensors(wl)
    for flags in (0, mvla.FLAG_INPUTS_STABLE):
        out = ctx.alloc_outputs(wl.samples, extras=True)
        for t in (out.out_hidden, out.out_k, out.out_v):
            t.view(torch.int16).fill_(0x5A5A)
        out.kept_idx.fill_(-77)
        ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"], flags=flags | mvla.FLAG_RESET_STATE,
                       out=out)
        torch.cuda.synchronize()
        n = out.total_kept
        assert 0 < n < out.kept_idx.numel() and int(out.out_offsets[-1]) == n
        assert bool((out.kept_idx[n:] == -77).all()), "list entries past the total were written"
        assert bool((out.kept_idx[:n] >= 0).all())
        for t in (out.out_hidden, out.out_k, out.out_v):
            assert bool((t[n:].view(torch.int16) == 0x5A5A).all()), "rows past the total were written"
    ctx.close()


def test_a_bounded_wait_that_runs_out_is_reported_and_sticky():
    # the wait is the one the row-copying CTAs use for a kept-list word; here it polls a word nothing sets,
    # with a limit of 200 us: the kernel ends by itself, the status word holds the error
    wl = W.small_workload(95, batch=1, D=256, H=2, d=64, dtype="bf16", n_txt=(5,), n_2d=(70,), n_3d=(150,))
    dev = device_tensors(wl)
    ctx = mvla.context_for(wl)
    ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])     # healthy before
    torch.cuda.synchronize()
    t0 = torch.cuda.Event(enable_timing=True); t1 = torch.cuda.Event(enable_timing=True)
    t0.record()
    ctx.selftest_wait_timeout(200)
    t1.record()
    torch.cuda.synchronize()
    assert 0.15 < t0.elapsed_time(t1) < 50.0, "the wait must end by itself after about its limit"
    for call in (lambda: ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"]),
                 lambda: ctx.salience(wl.samples, dev["q"], dev["k"])):
        with pytest.raises(mvla.MvlaError) as e:
            call()
        assert e.value.code == mvla.ERR_TIMEOUT                       # sticky: every later call reports it
    ctx.close()
    ctx2 = mvla.context_for(wl)                                       # a fresh context works
    out, refs = run_and_check_step(ctx2, wl, 0, _fresh_states(wl))
    with pytest.raises(mvla.MvlaError) as e:
        ctx2.selftest_wait_timeout(0)                                 # the limit must be 1 us .. 1 s
    assert e.value.code == mvla.ERR_INVALID_ARG
    ctx2.close()


# ------------------------------------------------------------------ reuse of the previous action step's logits
@pytest.mark.parametrize("drift,T", [("all", 16), ("visual_local", 8)])
def test_action_iteration_reusing_the_previous_steps_logits(drift, T):
    # every step is judged against the FULL oracle on the step's own inputs: with a truthful mask the reuse
    # must not be visible in the results
    wl = W.config5_action_iteration(T=T, drift=drift)
    ctx = mvla.context_for(wl, logit_cache=1)
    states = _fresh_states(wl)
    per_step = []
    for t in range(T):
        before = ctx.logit_cache_stats()
        run_and_check_step(ctx, wl, t, states, flags=mvla.FLAG_RESET_STATE if t == 0 else 0,
                           changed_rows=wl.extra["changed_rows"][t] if t > 0 else None)
        after = ctx.logit_cache_stats()
        per_step.append((after[0] - before[0], after[1] - before[1]))
    assert per_step[0] == (10, 0)                                     # 2 image + 8 point tiles, nothing to reuse yet
    assert all(c + r == 10 for c, r in per_step)
    if drift == "visual_local":                                       # one run of 131 rows: two or three tiles change
        assert all(1 <= c <= 3 for c, r in per_step[1:])
    ctx.close()


def test_a_mask_that_hides_a_change_reuses_the_stale_logits():
    # shows that the cache is what is read: with a mask that claims nothing changed, step 2 returns step 1's scores
    wl = W.config5_action_iteration(T=2, D=256, H=4, d=64, n_txt=20, n_2d=150, n_3d=300, drift="visual_local")
    ctx = mvla.context_for(wl, logit_cache=1)
    wl.steps[1].k[:40] *= np.float32(-2.0)                            # a change no tolerance can hide (exact in bf16)
    dev0, dev1 = device_tensors(wl, 0), device_tensors(wl, 1)
    out0 = ctx.prune_step(0, wl.samples, wl.mode, dev0["q"], dev0["k"], dev0["v"], dev0["hidden"], flags=mvla.FLAG_RESET_STATE)
    attn0 = out0.attn.clone()
    lie = np.zeros(wl.samples[0].seq_len, dtype=np.uint8)
    out1 = ctx.prune_step(0, wl.samples, wl.mode, dev1["q"], dev1["k"], dev1["v"], dev1["hidden"], changed_rows=lie)
    torch.cuda.synchronize()
    assert torch.equal(out1.attn, attn0)
    t1 = wl.steps[1]
    truth = oracle.salience(t1.q, t1.k, wl.n_heads, wl.head_dim, wl.samples[0])
    got = out1.attn.cpu().numpy()
    assert (np.abs(got - truth) > 20 * SALIENCE_RTOL * np.abs(truth)).sum() >= 20, "the stale logits were not what was used"
    # and with the truthful mask the same step is right
    ctx.prune_step(0, wl.samples, wl.mode, dev0["q"], dev0["k"], dev0["v"], dev0["hidden"], flags=mvla.FLAG_RESET_STATE)
    out2 = ctx.prune_step(0, wl.samples, wl.mode, dev1["q"], dev1["k"], dev1["v"], dev1["hidden"],
                          changed_rows=wl.extra["changed_rows"][1] | (np.arange(wl.samples[0].seq_len) < 40))
    torch.cuda.synchronize()
    assert_salience_close(out2.attn.cpu().numpy(), truth)
    assert ctx.logit_cache_stats()[1] >= 5                            # step 2 reused all 2 + 3 tiles of step 1
    ctx.close()


def test_logit_cache_is_left_out_of_samples_that_its_kernel_does_not_take():
    # 9 + 8 key tiles in 2000 tokens: one tile more than the kernel that keeps logits covers.  Nothing is reused or counted,
    # whatever the mask says, and every step is judged against the full oracle on its own inputs
    wl = W.config5_action_iteration(T=3, D=256, H=4, d=64, n_txt=20, n_2d=1100, n_3d=900, drift="visual_local")
    ctx = mvla.context_for(wl, logit_cache=1)
    states = _fresh_states(wl)
    for t in range(3):
        run_and_check_step(ctx, wl, t, states, flags=mvla.FLAG_RESET_STATE if t == 0 else 0,
                           changed_rows=wl.extra["changed_rows"][t] if t > 0 else None)
        assert ctx.logit_cache_stats() == (0, 0)
    ctx.close()


def test_a_step_beside_a_sample_without_logit_cache_leaves_no_logits_to_reuse():
    # the small sample (2 + 3 tiles) is stepped beside one of 17 tiles, then alone with a mask, then alone once more
    wl = W.small_workload(83, batch=2, D=256, H=4, d=64, n_txt=(20, 30), n_2d=(150, 1100), n_3d=(300, 900))
    ctx, small, t = mvla.context_for(wl, logit_cache=1), wl.samples[0], wl.steps[0]
    dev = device_tensors(wl)
    ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"], flags=mvla.FLAG_RESET_STATE)
    assert ctx.logit_cache_stats() == (0, 0)
    for computed, reused in ((5, 0), (6, 4)):
        mask = np.zeros(wl.total_rows, dtype=np.uint8)
        mask[small.seq_off + small.off_2d:][:40] = 1
        t.k[mask != 0] *= np.float32(-2.0)                            # (exact in bf16)
        k = mvla.to_device(t.k, wl.dtype, "cuda")
        out = ctx.prune_step(0, [small], wl.mode, dev["q"], k, dev["v"], dev["hidden"], changed_rows=mask)
        torch.cuda.synchronize()
        assert_salience_close(out.attn.cpu().numpy(), oracle.salience(t.q, t.k, wl.n_heads, wl.head_dim, small))
        assert ctx.logit_cache_stats() == (computed, reused)
    ctx.close()


def test_a_step_through_the_stage_calls_makes_the_cached_logits_stale():
    # step 2 runs as salience + select: a mask for step 3 says what changed since step 2, and the cache holds step 1
    wl = W.config5_action_iteration(T=1, D=256, H=4, d=64, n_txt=20, n_2d=150, n_3d=300)
    ctx, s, t, dev = mvla.context_for(wl, logit_cache=1), wl.samples[0], wl.steps[0], device_tensors(wl)
    ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"], flags=mvla.FLAG_RESET_STATE)
    t.k[s.off_2d:s.off_2d + 40] *= np.float32(-2.0)                   # (exact in bf16)
    k = mvla.to_device(t.k, wl.dtype, "cuda")
    attn, l1 = ctx.salience(wl.samples, dev["q"], k, dev["hidden"])
    ctx.select(0, wl.samples, wl.mode, attn, l1)
    nothing = np.zeros(s.seq_len, dtype=np.uint8)
    out = ctx.prune_step(0, wl.samples, wl.mode, dev["q"], k, dev["v"], dev["hidden"], changed_rows=nothing)
    torch.cuda.synchronize()
    assert_salience_close(out.attn.cpu().numpy(), oracle.salience(t.q, t.k, wl.n_heads, wl.head_dim, s))
    assert ctx.logit_cache_stats() == (10, 0)
    ctx.close()


@pytest.mark.parametrize("n_txt,n_2d,n_3d", [(40, 700, 900), (64, 512, 640), (17, 1500, 500), (48, 100, 60)])
def test_step_with_two_threads_per_key_in_every_shape_of_the_scoring_kernel(n_txt, n_2d, n_3d):
    # more than 16 text queries: the scoring kernel of the fused step runs with two threads per key, half of the
    # queries each; 33-64 queries use 64 tensor-memory columns (the second half partly empty at 40 and 48), more
    # than 1024 visual tokens put two key tiles on a CTA
    wl = W.small_workload(97, batch=1, D=128, H=2, d=64, dtype="bf16", n_txt=(n_txt,), n_2d=(n_2d,), n_3d=(n_3d,),
                          keep=(0.4,), steps=2)
    ctx = mvla.context_for(wl)
    states = _fresh_states(wl)
    for t in range(2):
        run_and_check_step(ctx, wl, t, states)
    ctx.close()


@pytest.mark.parametrize("batch,H,n_txt,n_2d,n_3d,kw", [
    (8, 16, (1, 16, 17, 64), (128, 129, 1), (255, 300, 513), {}),            # every padded text length; ragged tiles of one key up
    (12, 16, (5, 9), (130, 40), (37, 200), {"dtype": "fp8"}),                # 8-bit keys, 16-query slots
    (10, 16, (33, 48), (256, 100), (129, 384), {"n_kv_heads": 4}),           # grouped key heads
    (9, 16, (40, 20), (200, 60), (70, 300), {"d": 96}),                      # a partial swizzle row
    (6, 8, (64, 3), (1000, 700), (900, 1047), {"d": 256}),                   # four stages per tile; clusters of two
    (1, 4, (64,), (2048,), (2048,), {"D": 512}),                             # the most tiles: clusters of eight
    (2, 4, (17, 50), (1500, 2000), (1200, 77), {"text_first": True})])       # more than 2048 tokens, 1024-thread tail
def test_streaming_scoring_kernel_at_the_edges_of_its_shapes(batch, H, n_txt, n_2d, n_3d, kw):
    """Batches whose CTAs do not all run at once, and samples of more than 16 key tiles, go through the streaming
    scoring kernel; two action steps, so that its ring state and the accumulators it leaves are exercised twice."""
    kw = {"D": 256, "d": 64, **kw}
    wl = W.small_workload(71, batch=batch, H=H, n_txt=n_txt, n_2d=n_2d, n_3d=n_3d, keep=(0.3, 0.5, 0.2), steps=2, **kw)
    ctx = mvla.context_for(wl)
    states = [oracle.State(s.n_vis) for s in wl.samples]
    for step in range(2):
        if "n_kv_heads" not in kw:
            run_and_check_step(ctx, wl, step, states)
            continue
        t, dev = wl.steps[step], device_tensors(wl, step)        # the oracle's step takes ungrouped keys: scores only
        out = ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])
        attn, vis = out.attn.cpu().numpy(), 0
        for s in wl.samples:
            assert_salience_close(attn[vis:vis + s.n_vis], oracle.salience_gqa(t.q, t.k, H, kw["n_kv_heads"], kw["d"], s))
            vis += s.n_vis
    ctx.close()


@pytest.mark.parametrize("D", [8, 2056, 4096, 4104])          # pieces of 8 KB a row: one of 16 bytes; a part; one; one and 16 bytes
@pytest.mark.parametrize("batch,H,n_txt,n_2d,n_3d,kw", [
    (8, 32, (5, 33, 64), (0, 200, 129, 1), (130, 64, 300, 90), {}),          # a modality without tokens; samples of a few rows
    (3, 64, (16, 48), (200, 256), (64, 77), {"dtype": "fp8", "text_first": True})])
def test_streaming_scoring_kernel_with_norms_inside(batch, H, n_txt, n_2d, n_3d, kw, D):
    """Adaptive batches have their feature norms taken by two warps of the scoring kernel: rows of every sample, in pieces that
    end anywhere; two action steps."""
    wl = W.small_workload(75, batch=batch, H=H, D=D, d=64, n_txt=n_txt, n_2d=n_2d, n_3d=n_3d, keep=(0.3, 0.5), steps=2, **{"dtype": "bf16", **kw})
    ctx, states = mvla.context_for(wl), [oracle.State(s.n_vis) for s in wl.samples]
    for step in range(2):
        run_and_check_step(ctx, wl, step, states)
    ctx.close()


@pytest.mark.parametrize("batch,H,n_txt,n_2d,n_3d", [
    (8, 16, (64, 1, 33), (129, 40), (255, 300)),
    (2, 4, (17, 50), (1500, 2000), (1200, 77))])
def test_streaming_scoring_kernel_without_norms_beside_it(batch, H, n_txt, n_2d, n_3d):
    """Fixed budgets need no feature norms: the kernel's other register split."""
    wl = W.small_workload(73, batch=batch, H=H, D=256, n_txt=n_txt, n_2d=n_2d, n_3d=n_3d, mode=W.MODE_FIXED, steps=2)
    ctx = mvla.context_for(wl)
    states = [oracle.State(s.n_vis) for s in wl.samples]
    for step in range(2):
        run_and_check_step(ctx, wl, step, states)
    ctx.close()


@pytest.mark.parametrize("batch,d,n_txt,n_2d,n_3d,mode,at_once", [
    (1, 256, 20, 768, 768, W.MODE_ADAPTIVE, True),        # 16 clusters of 6 CTAs with two tiles, one CTA to a multiprocessor
    (1, 256, 20, 768, 1023, W.MODE_ADAPTIVE, False),      # 16 of 7: one more than lie inside the device's GPCs
    (1, 128, 64, 768, 1023, W.MODE_ADAPTIVE, True),       # rows half as long: two CTAs fit
    (1, 160, 64, 1023, 1000, W.MODE_ADAPTIVE, False),     # 16 of 8, rows of one and a quarter boxes
    (2, 256, 7, 640, 512, W.MODE_FIXED, False),           # 32 of 5
    (4, 256, 33, 256, 512, W.MODE_FIXED, False),          # 384 CTAs of one tile, two fit: 296 at once
    (4, 256, 33, 256, 512, W.MODE_ADAPTIVE, True),        # ... with norms beside the scores the line is three to a multiprocessor
    (4, 128, 33, 256, 512, W.MODE_FIXED, True),           # ... and three fit
])
def test_scoring_kernel_goes_by_what_fits_on_the_device(batch, d, n_txt, n_2d, n_3d, mode, at_once):
    """16 heads on both sides of the line between the two scoring kernels, told apart by how many CTAs leave time stamps:
    the latency-shaped kernel has one per one or two key tiles."""
    wl = W.small_workload(74, batch=batch, D=128, H=16, d=d, n_txt=(n_txt,), n_2d=(n_2d,), n_3d=(n_3d,), keep=(0.3,), mode=mode, steps=2)
    ctx, states = mvla.context_for(wl), [oracle.State(s.n_vis) for s in wl.samples]
    tiles = -(-n_2d // 128) + -(-n_3d // 128)
    ctas = batch * 16 * -(-tiles // -(-tiles // 8))
    for step in range(2):
        stamps = torch.zeros(2, ctx.STAMP_SLOTS, 2, dtype=torch.int64, device="cuda")
        ctx.set_kernel_stamps(stamps)
        run_and_check_step(ctx, wl, step, states)
        assert (int((stamps[0, :, 1] != 0).sum()) == ctas) == at_once
    ctx.close()


@pytest.mark.parametrize("batch,H,n_txt,n_2d,n_3d,kw,beside", [
    (13, 24, (33, 16, 64), (256, 300, 1), (400, 384, 700), {}, True),                       # one tile of one token; three rounds of jobs
    (13, 24, (33, 16, 64), (256, 300, 1), (400, 384, 700), {"text": "middle"}, True),       # rows of the text known with the list only
    (13, 24, (5, 17), (300, 0), (400, 700), {"mode": W.MODE_FIXED, "text_first": True}, True),   # no norms; a modality without tokens
    (13, 24, (33, 64), (256, 300), (400, 384), {"cold_start": 1}, True),                     # all kept first: norms after the list
    (13, 24, (33, 64), (200, 160), (380, 440), {}, False),                                   # keys of a job below the line
    (12, 24, (33, 64), (256, 300), (400, 384), {}, False),                                   # two rounds
    (36, 24, (3, 20), (256, 300), (400, 384), {}, True),                                     # a launch of 32 samples beside, one of 4 (96 CTAs) behind
    (7, 24, (64, 50), (600, 300), (500, 1024), {}, True),                                    # clusters of two, up to 1324 tokens
    (3, 24, (64, 50), (1500, 900), (700, 1300), {}, True)])                                  # clusters of four, 2200 tokens
def test_tail_beside_the_streaming_scoring_kernel(batch, H, n_txt, n_2d, n_3d, kw, beside):
    """Batches whose samples are selected and copied while others are scored, told by the multiprocessors that the scoring kernel leaves
    free; two action steps, the same bits when they are run again."""
    kw = dict(kw)
    text = kw.pop("text", "")
    wl = W.small_workload(76, batch=batch, H=H, D=128, d=128, n_txt=n_txt, n_2d=n_2d, n_3d=n_3d, keep=(0.3, 0.5), steps=2, **kw)
    if text == "middle":
        wl.samples[:] = [W.Sample(**{**vars(s), "off_2d": 0, "off_txt": s.n_2d, "off_3d": s.n_2d + s.n_txt}) for s in wl.samples]
    ctx, states = mvla.context_for(wl), [oracle.State(s.n_vis) for s in wl.samples]
    for step in range(2):
        stamps = torch.zeros(2, ctx.STAMP_SLOTS, 2, dtype=torch.int64, device="cuda")
        ctx.set_kernel_stamps(stamps)
        run_and_check_step(ctx, wl, step, states)
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert (int((stamps[0, :, 1] != 0).sum()) <= sms - 12 and int((stamps[1, :, 0] != 0).sum()) >= sms) == beside
    ctx.set_kernel_stamps(None)
    dev, runs = device_tensors(wl), []
    for _ in range(8):
        out = ctx.alloc_outputs(wl.samples, extras=True)
        ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"], flags=mvla.FLAG_RESET_STATE, out=out)
        n = int(out.out_offsets[-1])
        runs.append([out.budgets, out.ahat] + [t[:n] for t in (out.kept_idx, out.out_hidden, out.out_k, out.out_v)])
    for r in runs[1:]:
        assert all(torch.equal(x.contiguous().view(torch.uint8), y.contiguous().view(torch.uint8)) for x, y in zip(runs[0], r))
    ctx.close()


FORMS = {                     # heads, head dim, key heads, dtype, hidden width, samples, text, 2D, 3D, mode
    "rows_of_two_pieces": (48, 128, 0, torch.bfloat16, 4104, 7, (33, 16, 64), (256, 300), (400, 384), mvla.MODE_ADAPTIVE),
    "heads_of_256": (16, 256, 0, torch.bfloat16, 512, 20, (64, 5), (120, 130), (210, 200), mvla.MODE_ADAPTIVE),       # a ring of five stages
    "e4m3": (48, 128, 0, torch.float8_e4m3fn, 264, 7, (16, 48), (600, 640), (700, 760), mvla.MODE_ADAPTIVE),
    "e4m3_grouped": (32, 128, 8, torch.float8_e4m3fn, 256, 10, (7, 16), (600, 640), (700, 760), mvla.MODE_FIXED),
    "grouped": (32, 128, 8, torch.bfloat16, 256, 10, (33, 64), (256, 300), (400, 384), mvla.MODE_FIXED),
    "one_key_head": (32, 128, 1, torch.bfloat16, 64, 10, (1, 64), (0, 300), (700, 384), mvla.MODE_FIXED),
    "above_2048_tokens": (24, 128, 0, torch.bfloat16, 128, 4, (48, 64), (100, 1500), (700, 1300), mvla.MODE_ADAPTIVE),   # CTAs of 32 warps; the last sample the longest
}


@pytest.mark.parametrize("outputs", ["all", "hidden", "none", "dry"])
@pytest.mark.parametrize("form", FORMS)
def test_tail_beside_gives_what_the_tail_behind_gives(form, outputs):
    """The same batches from a tail beside the scoring kernel, from one behind it (an event set between the kernels) and from a graph that is replayed:
    the same bits; the indicators, whose norms other warps have summed, to the last few bits of fp32."""
    H, d, hkv, dtype, D, batch, n_txt, n_2d, n_3d, mode = FORMS[form]
    samples, off = [], 0
    for b in range(batch):
        s = W.layout_2d_3d_txt(off, n_txt[b % len(n_txt)], n_2d[b % len(n_2d)], n_3d[b % len(n_3d)], keep_2d=0.3, keep_3d=0.4, keep_total=(0.2, 0.5)[b % 2], state_slot=b)
        samples.append(s)
        off += s.seq_len
    gen = torch.Generator(device="cuda").manual_seed(81)
    draw = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    q, k, v = (draw(off, h, d).to(dtype) for h in (H, hkv or H, hkv or H))
    hidden = draw(off, D).to(torch.bfloat16)
    ctx = mvla.PruneContext(dtype=dtype, n_heads=H, head_dim=d, d_model=D, max_batch=batch, max_text=64, max_2d=max(n_2d), max_3d=max(n_3d), n_kv_heads=hkv,
                            cold_start_full_keep=0, tau_2d=0.35, tau_3d=0.65)
    flags = mvla.FLAG_RESET_STATE | (mvla.FLAG_NO_STATE_UPDATE if outputs == "dry" else 0)

    def fresh():
        out = ctx.alloc_outputs(samples, hidden=outputs != "none", kv=outputs in ("all", "dry"), extras=True)
        for t in vars(out).values():
            if torch.is_tensor(t):
                t.view(torch.uint8).zero_()
        return out
    call = lambda out: ctx.prune_step(0, samples, mode, q, k, v if out.out_v is not None else None, hidden, flags=flags, out=out)
    stamps = torch.zeros(2, ctx.STAMP_SLOTS, 2, dtype=torch.int64, device="cuda")
    ctx.set_kernel_stamps(stamps)
    sms, event = torch.cuda.get_device_properties(0).multi_processor_count, torch.cuda.Event()
    beside, behind = fresh(), fresh()
    call(beside)
    assert int((stamps[0, :, 1] != 0).sum()) <= sms - 12 and int((stamps[1, :, 0] != 0).sum()) >= (sms if outputs != "none" else 1)
    event.record()
    ctx.set_stage_event(event)
    call(behind)
    ctx.set_stage_event(None)
    ctx.set_kernel_stamps(None)
    captured, graph = fresh(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(7):                                # the rotation of scratch sets comes round
            call(captured)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for out in (behind, captured):
        for name, t in vars(beside).items():
            other = getattr(out, name)
            if name == "diag":
                a, b = t.cpu().numpy(), other.cpu().numpy()
                assert np.array_equal(a[:, :7], b[:, :7])
                np.testing.assert_allclose(b[:, 8:].copy().view(np.float32), a[:, 8:].copy().view(np.float32), rtol=2e-6)
            elif torch.is_tensor(t):
                assert torch.equal(t.view(torch.uint8), other.view(torch.uint8)), name
    ctx.close()


def test_an_event_between_the_kernels_keeps_the_tail_behind_the_scoring_kernel():
    """With a stage event set, a batch whose tail would run beside its scoring kernel is scored on all multiprocessors, and no copying
    CTA starts before the last scoring CTA has ended."""
    wl = W.small_workload(77, batch=13, H=24, D=128, d=128, n_txt=(33, 16, 64), n_2d=(256, 300), n_3d=(400, 384), keep=(0.3, 0.5), steps=2)
    ctx, states = mvla.context_for(wl), [oracle.State(s.n_vis) for s in wl.samples]
    event = torch.cuda.Event(enable_timing=True)
    event.record()
    ctx.set_stage_event(event)
    for step in range(2):
        stamps = torch.zeros(2, ctx.STAMP_SLOTS, 2, dtype=torch.int64, device="cuda")
        ctx.set_kernel_stamps(stamps)
        run_and_check_step(ctx, wl, step, states)
        scored, copied = stamps[0, :, 1], stamps[1, len(wl.samples):, 0]
        assert int((scored != 0).sum()) == torch.cuda.get_device_properties(0).multi_processor_count
        assert int(copied[copied != 0].min()) >= int(scored.max())
    ctx.close()


@pytest.mark.parametrize("batch,n_txt,n_2d,n_3d", [(13, (33, 16, 64), (256, 300), (400, 384)), (2, (12, 30), (100, 256), (300, 140))])
def test_live_steps_with_captured_steps_between_them_in_the_rotation_of_scratch_sets(batch, n_txt, n_2d, n_3d):
    """Two steps queued behind other work of their stream, and five that are captured in between: the second one comes round to the scratch
    set of the first."""
    wl = W.small_workload(80, batch=batch, H=24, D=128, d=128, n_txt=n_txt, n_2d=n_2d, n_3d=n_3d, keep=(0.3, 0.5), cold_start=0)
    ctx, dev = mvla.context_for(wl), device_tensors(wl)
    outs = [ctx.alloc_outputs(wl.samples, extras=True) for _ in range(4)]
    call = lambda out: ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"], flags=mvla.FLAG_RESET_STATE, out=out)
    live, side, graph = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    call(outs[0])
    torch.cuda.synchronize()
    with torch.cuda.stream(live):
        torch.cuda._sleep(20_000_000)                     # some 10 ms: the steps below wait in line, one behind the other
        call(outs[1])
    with torch.cuda.stream(side):
        graph.capture_begin(capture_error_mode="relaxed")
        for _ in range(5):
            call(outs[2])
        graph.capture_end()
    with torch.cuda.stream(live):
        call(outs[3])
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    n = int(outs[0].out_offsets[-1])
    for out in outs[1:]:
        assert torch.equal(out.budgets, outs[0].budgets) and torch.equal(out.ahat, outs[0].ahat)
        for name in ("kept_idx", "out_hidden", "out_k", "out_v"):
            assert torch.equal(getattr(out, name)[:n], getattr(outs[0], name)[:n]), name
    call(outs[1])                                         # no wait ran out
    torch.cuda.synchronize()
    ctx.close()


def test_stamps_of_a_tail_beside_the_scoring_kernel():
    """Selecting CTAs report the time of their last list as start and end; copying CTAs start before the scoring kernel has ended."""
    wl = W.small_workload(79, batch=13, H=24, D=128, d=128, n_txt=(33, 16, 64), n_2d=(256, 300), n_3d=(400, 384), keep=(0.3, 0.5), cold_start=0)
    ctx, stamps = mvla.context_for(wl), torch.zeros(2, mvla.PruneContext.STAMP_SLOTS, 2, dtype=torch.int64, device="cuda")
    ctx.set_kernel_stamps(stamps)
    run_and_check_step(ctx, wl, 0, [oracle.State(s.n_vis) for s in wl.samples])
    scored, tail = stamps[0].cpu(), stamps[1].cpu()
    tail = tail[tail[:, 1] != 0]
    selecting = tail[:, 0] == tail[:, 1]
    n = int(selecting.sum())
    assert 1 <= n <= 8 and selecting[:n].all() and (tail[n:, 0] < tail[n:, 1]).all() and (tail[:, 0] > 0).all()
    assert tail[n:, 0].min() < scored[:, 1].max() < tail[:n, 1].max()
    ctx.close()


def test_outputs_in_the_memory_of_the_queries_are_written_when_all_samples_are_scored():
    """Positions and smoothed scores that a caller has written over its queries: the same as in buffers of their own, from a tail that starts
    behind the scoring kernel."""
    wl = W.small_workload(78, batch=13, H=24, D=128, d=128, n_txt=(33, 16, 64), n_2d=(256, 300), n_3d=(400, 384), keep=(0.3, 0.5), cold_start=0)
    ctx, dev = mvla.context_for(wl), device_tensors(wl)
    call = lambda out: ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"], flags=mvla.FLAG_RESET_STATE, out=out)
    ref = call(ctx.alloc_outputs(wl.samples, extras=True))
    torch.cuda.synchronize()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for name in ("kept_idx", "ahat"):
        out = ctx.alloc_outputs(wl.samples, extras=True)
        keep = dev["q"].clone()
        own = getattr(out, name)
        setattr(out, name, dev["q"].view(-1)[-2 * own.numel():].view(own.dtype))     # the queries of the last samples
        stamps = torch.zeros(2, ctx.STAMP_SLOTS, 2, dtype=torch.int64, device="cuda")
        ctx.set_kernel_stamps(stamps)
        call(out)
        torch.cuda.synchronize()
        n = int(ref.out_offsets[-1])
        assert int((stamps[0, :, 1] != 0).sum()) == sms
        assert torch.equal(out.kept_idx[:n], ref.kept_idx[:n]) and torch.equal(out.ahat, ref.ahat) and torch.equal(out.out_v[:n], ref.out_v[:n])
        dev["q"].copy_(keep)
    ctx.close()


@pytest.mark.parametrize("gain", [30.0, 300.0])
def test_streaming_scoring_kernel_moves_its_references_when_exponents_would_overflow(gain):
    """Keys whose logits grow from tile to tile by far more than an fp32 exponent holds."""
    wl = W.small_workload(72, batch=10, D=256, H=16, d=64, n_txt=(20, 33), n_2d=(300, 128), n_3d=(260, 400))
    t = wl.steps[0]
    for s in wl.samples:
        for off, n in ((s.off_2d, s.n_2d), (s.off_3d, s.n_3d)):
            k = t.k[s.seq_off + off: s.seq_off + off + n]
            k *= (1.0 + gain * (np.arange(n) // 128)).astype(np.float32)[:, None, None]
    t.k[:] = W.round_to_dtype(t.k, "bf16")
    ctx, dev = mvla.context_for(wl), device_tensors(wl)
    out = ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])
    attn, vis = out.attn.cpu().numpy(), 0
    for s in wl.samples:
        assert_salience_close(attn[vis:vis + s.n_vis], oracle.salience_gqa(t.q, t.k, 16, 16, 64, s))
        vis += s.n_vis
    ctx.close()


@pytest.mark.parametrize("n_txt,n_2d,n_3d,d,hkv", [
    ((1, 17), (128, 1), (129, 40), 64, 0),                # one query, one key in a tile
    ((33, 64), (100, 256), (300, 0), 128, 2),             # both halves of the queries; an empty modality; grouped keys
    ((16, 48), (700, 513), (500, 640), 96, 0),            # two key tiles per CTA
    ((20, 5), (130, 60), (200, 90), 256, 0)])             # the longest rows
def test_fp32_step_at_the_edges_of_its_scoring_kernel(n_txt, n_2d, n_3d, d, hkv):
    wl = W.small_workload(73, batch=2, D=256, H=4, d=d, dtype="fp32", n_txt=n_txt, n_2d=n_2d, n_3d=n_3d, n_kv_heads=hkv)
    ctx, dev, t = mvla.context_for(wl), device_tensors(wl), wl.steps[0]
    if not hkv:
        run_and_check_step(ctx, wl, 0, [oracle.State(s.n_vis) for s in wl.samples])
    else:
        out = ctx.prune_step(0, wl.samples, wl.mode, dev["q"], dev["k"], dev["v"], dev["hidden"])
        attn, vis = out.attn.cpu().numpy(), 0
        for s in wl.samples:
            assert_salience_close(attn[vis:vis + s.n_vis], oracle.salience_gqa(t.q, t.k, 4, hkv, d, s))
            vis += s.n_vis
    ctx.close()
