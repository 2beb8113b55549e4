"""Behaviour of the C ABI on a GPU beyond plain parity: host-buffer step, call-order errors,
context reuse, bookkeeping queries, profiling counters, schedule variants."""
import numpy as np
import pytest
import torch

from paper_2412_20105_b200 import binding as B
from synth import SynthInputs, get_workload
from gpu_harness import GpuRun, run_and_check
from helpers import make_schedule

pytestmark = pytest.mark.gpu


def _small(**kw):
    base = dict(dtype="bf16", head_dim=128, num_heads=4, num_layers=6, batch=2, sys_len=5, num_visual=200,
                text_len_min=3, text_len_max=20, decode_steps=12, first_prune_layer=2, stride=2,
                step_ratio_bp=1500, tau=12.0, num_planted=10)
    base.update(kw)
    return get_workload("tiny").scaled(**base)


@pytest.mark.parametrize("packed", [False, True])
def test_host_buffer_step_equals_device_step(packed):
    """`packed`: q, k_new, v_new back to back in one pinned buffer (the library's single-copy path);
    otherwise three separate buffers (three copies)."""
    wl = _small()
    a, b = GpuRun(wl), GpuRun(wl)
    try:
        a.prefill(); b.prefill()
        assert torch.equal(a.out, b.out)
        for t in range(1, 6):
            a.decode(t)
            q, kn, vn = b.inputs(t)
            if packed:
                hqkv = torch.stack([q.cpu(), kn.cpu(), vn.cpu()]).contiguous().pin_memory()
                hq, hk, hv = hqkv[0], hqkv[1], hqkv[2]
                assert hk.data_ptr() == hq.data_ptr() + hq.numel() * hq.element_size()
            else:
                hq, hk, hv = (x.cpu().pin_memory() for x in (q, kn, vn))
            hout = torch.empty_like(q.cpu()).pin_memory()
            b.ctx.decode_step_host(t, hq, hk, hv, hout)
            torch.cuda.synchronize()
            assert torch.equal(hout, a.out.cpu()), t
            for l in range(wl.num_layers):
                ia, ca, _ = a.kept(l)
                ib, cb, _ = b.kept(l)
                assert np.array_equal(ca, cb)
                for s in range(wl.batch):
                    assert np.array_equal(ia[s, :ca[s]], ib[s, :cb[s]])
        assert a.ctx.status() == 0 and b.ctx.status() == 0
    finally:
        a.close(); b.close()


@pytest.mark.parametrize("overlap", [False, True])
def test_host_buffer_generation_runs_ahead_of_the_gpu(overlap):
    """Prefill and every decode step through the host-buffer calls, enqueued back to back with no synchronisation
    in between (the library's copy streams run ahead of and behind the kernels), against the same generation
    with device buffers: outputs bit-identical, same kept ids.  st3_host_sync + a wait on the caller's stream
    is all that makes the host outputs readable."""
    wl = _small()
    steps = 9
    a, b = GpuRun(wl), GpuRun(wl, overlap=overlap, host_prefill=1)
    try:
        g = b.g
        q0 = g.queries([0])[0]
        K, V = g.prompt_kv(range(wl.num_layers))
        hq0, hK, hV = q0.pin_memory(), K.pin_memory(), V.pin_memory()
        hout0 = torch.empty_like(hq0).pin_memory()
        qs = g.queries(list(range(1, steps + 1)))
        kn, vn = g.new_kv(list(range(1, steps + 1)))
        hqkv = torch.stack([qs, kn, vn], dim=1).contiguous().pin_memory()        # [step][q | k | v]
        hout = torch.zeros_like(qs).pin_memory()
        b.ctx.prefill_select_host(hq0, hK, hV, g.text_len.tolist(), hout0)
        for t in range(1, steps + 1):
            b.ctx.decode_step_host(t, hqkv[t - 1, 0], hqkv[t - 1, 1], hqkv[t - 1, 2], hout[t - 1])
        b.ctx.host_sync()
        torch.cuda.current_stream().synchronize()
        a.prefill()
        assert torch.equal(hout0, a.out.cpu())
        for t in range(1, steps + 1):
            a.decode(t)
            assert torch.equal(hout[t - 1], a.out.cpu()), t
        for l in range(wl.num_layers):
            ia, ca, _ = a.kept(l)
            ib, cb, _ = b.kept(l)
            assert np.array_equal(ca, cb)
            for s in range(wl.batch):
                assert np.array_equal(ia[s, :ca[s]], ib[s, :cb[s]])
        assert a.ctx.status() == 0 and b.ctx.status() == 0
        # a second generation on the same context reuses the staging areas behind the first one's work
        b.ctx.prefill_select_host(hq0, hK, hV, g.text_len.tolist(), hout0)
        b.ctx.decode_step_host(1, hqkv[0, 0], hqkv[0, 1], hqkv[0, 2], hout[0])
        b.ctx.host_sync()
        torch.cuda.current_stream().synchronize()
        a.prefill(); a.decode(1)
        assert torch.equal(hout[0], a.out.cpu()) and b.ctx.status() == 0
    finally:
        a.close(); b.close()


def test_host_buffer_prefill_needs_its_staging_areas():
    wl = _small()
    run = GpuRun(wl)                       # host_prefill = 0
    try:
        g = run.g
        q0 = g.queries([0])[0].pin_memory()
        K, V = g.prompt_kv(range(wl.num_layers))
        with pytest.raises(B.St3Error) as e:
            run.ctx.prefill_select_host(q0, K.pin_memory(), V.pin_memory(), g.text_len.tolist(),
                                        torch.empty_like(q0).pin_memory())
        assert e.value.code == 3
    finally:
        run.close()


def test_call_order_and_capacity_errors():
    wl = _small()
    run = GpuRun(wl)
    try:
        q, kn, vn = run.inputs(1)
        with pytest.raises(B.St3Error) as e:                      # decode before any prefill
            run.ctx.decode_step(1, q, kn, vn, run.out)
        assert e.value.code == 3
        run.prefill()
        with pytest.raises(B.St3Error) as e:                      # step gap
            run.ctx.decode_step(2, q, kn, vn, run.out)
        assert e.value.code == 3
        run.ctx.decode_step(1, q, kn, vn, run.out)
        with pytest.raises(B.St3Error) as e:                      # same step twice
            run.ctx.decode_step(1, q, kn, vn, run.out)
        assert e.value.code == 3
        with pytest.raises(B.St3Error) as e:                      # beyond max_decode_steps
            run.ctx.decode_step(wl.decode_steps + 1, q, kn, vn, run.out)
        assert e.value.code == 4
        with pytest.raises(B.St3Error) as e:                      # layer range out of bounds
            run.ctx.decode_step(2, q, kn, vn, run.out, layer_begin=1)
        assert e.value.code == 1
        with pytest.raises(B.St3Error) as e:                      # text longer than the configured maximum
            B.st3_prefill_select(run.ctx.handle, 0, wl.num_layers, run.q_cur.data_ptr(), run.q_cur.data_ptr(),
                                 run.q_cur.data_ptr(), [wl.text_len_max + 1] * wl.batch, run.out.data_ptr(), 0)
        assert e.value.code == 4
        with pytest.raises(B.St3Error) as e:                      # misaligned pointer
            B.st3_decode_step(run.ctx.handle, 2, 0, wl.num_layers, q.data_ptr() + 2, kn.data_ptr(), vn.data_ptr(),
                              run.out.data_ptr(), 0)
        assert e.value.code == 1
        # the failed calls changed nothing: step 2 still works and still matches the oracle
        before = run.snapshot(range(wl.num_layers))
        run.decode(2)
        for l in range(wl.num_layers):
            run.check_decode_unit(0, l, 2, before[l])
        assert run.ctx.status() == 0
    finally:
        run.close()


def test_context_is_reusable_for_a_new_generation():
    wl = _small()
    run = GpuRun(wl)
    try:
        run.prefill()
        for t in range(1, 5):
            run.decode(t)
        first = {l: run.kept(l) for l in range(wl.num_layers)}
        out_first = run.out.clone()
        run.prefill()                                             # same prompt again: state starts over
        for t in range(1, 5):
            run.decode(t)
        assert torch.equal(out_first, run.out)
        for l in range(wl.num_layers):
            ids, cnt, _ = run.kept(l)
            assert np.array_equal(cnt, first[l][1])
            for s in range(wl.batch):
                assert np.array_equal(ids[s, :cnt[s]], first[l][0][s, :cnt[s]])
        assert run.ctx.status() == 0
    finally:
        run.close()


def test_rows_held_and_launch_counters_follow_the_schedule():
    wl = _small()
    run = GpuRun(wl)
    try:
        assert run.ctx.rows_held() == (0, 0)
        n0 = run.ctx.launch_count()
        run.prefill()
        assert run.ctx.launch_count() - n0 == 3                   # attend, finish, gather
        sched = make_schedule(wl)
        text = run.g.text_len
        for t in range(0, 4):
            if t:
                run.decode(t)
            vis, oth = run.ctx.rows_held()
            assert vis == wl.batch * sum(sched.n(l, t) for l in range(wl.num_layers))
            assert oth == wl.num_layers * sum(wl.sys_len + int(x) + t for x in text)
        assert run.ctx.launch_count() - n0 == 3 + 2 * 3
        B.st3_profile_enable(run.ctx.handle, True)
        run.decode(4); run.decode(5)
        a_ms, f_ms, na, nf = B.st3_profile_read(run.ctx.handle)
        assert na == nf == 2 and a_ms > 0 and f_ms > 0
        B.st3_profile_enable(run.ctx.handle, False)
        assert run.ctx.status() == 0
    finally:
        run.close()


@pytest.mark.parametrize("anneal,kw", [("linear", dict(tau=12.0)), ("exp", dict(sigma=4.0)), ("none", dict())])
def test_other_attenuation_functions(anneal, kw):
    code = {"linear": B.ST3_ANNEAL_LINEAR, "exp": B.ST3_ANNEAL_EXP, "none": B.ST3_ANNEAL_NONE}[anneal]
    wl = _small(**{k: v for k, v in kw.items() if k == "tau"})
    stats = run_and_check(wl, wl.decode_steps, sched_kw=dict(anneal=anneal, **{k: v for k, v in kw.items() if k == "sigma"}),
                          anneal=code, **{k: v for k, v in kw.items() if k == "sigma"})
    assert stats["units"] == (wl.decode_steps + 1) * wl.num_layers * wl.batch


def test_layer_by_layer_calls_match_one_call_for_all_layers():
    wl = _small()
    a, b = GpuRun(wl), GpuRun(wl)
    try:
        a.prefill(); b.prefill(layers_per_call=1)
        assert torch.equal(a.out, b.out)
        for t in range(1, 5):
            a.decode(t); b.decode(t, layers_per_call=1)
            assert torch.equal(a.out, b.out), t
        assert a.ctx.status() == 0 and b.ctx.status() == 0
    finally:
        a.close(); b.close()


def _handmade(nv, H=2, D=64, sys_len=2, text=3, steps=4, keep_bp=5000, dtype="f32", **cfg_kw):
    cfg = B.make_config(num_layers=1, num_heads=H, head_dim=D, dtype=dtype, batch=1, sys_len=sys_len,
                        num_visual=nv, max_text_len=text, max_decode_steps=steps, stride=1, step_ratio_bp=0,
                        first_prune_layer=0, first_ratio_bp=10000 - keep_bp, tau=float(steps), **cfg_kw)
    return cfg, B.Context(cfg)


@pytest.mark.parametrize("static_rank", [0, 1])
def test_equal_scores_keep_the_lowest_original_indices(static_rank):
    """Every visual key identical => every visual score identical: Top must fall back on the index."""
    nv, H, D, sys_len, text = 200, 2, 64, 2, 3
    cfg, ctx = _handmade(nv, H, D, sys_len, text, static_rank=static_rank)
    try:
        g = torch.Generator().manual_seed(5)
        T0 = sys_len + nv + text
        K = torch.randn(1, 1, H, T0, D, generator=g)
        V = torch.randn(1, 1, H, T0, D, generator=g)
        K[:, :, :, sys_len:sys_len + nv] = K[:, :, :, sys_len:sys_len + 1]          # all visual keys alike
        q = torch.randn(1, 1, H, D, generator=g)
        out = torch.empty(1, 1, H, D, device="cuda")
        ctx.prefill_select(q.cuda(), K.cuda(), V.cuda(), [text], out)
        ids, cnt, mass = ctx.get_kept(0)
        n = int(cnt[0])
        assert n == nv // 2
        assert sorted(ids[0, :n].tolist()) == list(range(n))                        # the n lowest indices
        if static_rank:
            assert ids[0, :n].tolist() == list(range(n))                            # and in index order
        m = mass[0].cpu().numpy()
        assert np.all(m == m[0]) and m[0] > 0                                       # bit-identical scores
        # decode steps keep dropping the highest remaining indices
        for t in range(1, 4):
            kn = torch.randn(1, 1, H, D, generator=g).cuda()
            ctx.decode_step(t, q.cuda(), kn, kn, out)
            ids, cnt, _ = ctx.get_kept(0)
            k = B.st3_schedule_count(cfg, 0, t)
            assert int(cnt[0]) == k and sorted(ids[0, :k].tolist()) == list(range(k))
        assert ctx.status() == 0
    finally:
        ctx.close()


def _check_tied_classes(ctx, cfg, keys, q, dtype, sys_len, text, classes):
    """Visual token i carries the key of class i % classes: tokens of a class must score alike to the last bit wherever
    they stand in the prompt or (once holes have been filled) in the cache, and lose by their index only."""
    H, D, nv = cfg.num_heads, cfg.head_dim, cfg.num_visual
    t = dict(f32=torch.float32, bf16=torch.bfloat16)[dtype]
    g = torch.Generator().manual_seed(nv)
    K, V = (torch.randn(1, 1, H, sys_len + nv + text, D, generator=g) for _ in range(2))
    K[0, 0, :, sys_len:sys_len + nv] = keys[:, torch.arange(nv) % classes]
    kn = torch.randn(1, 1, H, D, generator=g).to(t).cuda()
    out = torch.empty(1, 1, H, D, dtype=t, device="cuda")
    vis = torch.arange(nv)
    for step in range(4):
        if step == 0:
            ctx.prefill_select(q[0].to(t).cuda(), K.to(t).cuda(), V.to(t).cuda(), [text], out)
        else:
            ctx.decode_step(step, q[step].to(t).cuda(), kn, kn, out)
        ids, cnt, mass = ctx.get_kept(0)
        mass = mass[0].cpu()
        k = B.st3_schedule_count(cfg, 0, step)
        for c in range(classes):
            m = mass[vis[vis % classes == c]]
            assert (m == m[:1]).all(), (step, c, m.unique().tolist())
        best = vis[np.lexsort((vis.numpy(), -mass[vis].numpy()))[:k]]
        assert int(cnt[0]) == k < len(vis) and sorted(ids[0, :k].tolist()) == sorted(best.tolist()), step
        vis = best.sort().values
    assert ctx.status() == 0


@pytest.mark.parametrize("dtype,D", [("f32", 64), ("f32", 128), ("bf16", 64), ("bf16", 128)])
@pytest.mark.parametrize("H", [1, 5])
def test_identical_keys_score_alike_wherever_they_stand(dtype, D, H):
    nv, sys_len, text = 333, 2, 3
    cfg, ctx = _handmade(nv, H, D, sys_len, text, steps=8, keep_bp=9000, dtype=dtype)
    try:
        g = torch.Generator().manual_seed(D + H)
        _check_tied_classes(ctx, cfg, torch.randn(H, 15, D, generator=g), torch.randn(4, 1, 1, H, D, generator=g), dtype,
                            sys_len, text, 15)
    finally:
        ctx.close()


def test_two_score_levels_with_ties_at_the_cut():
    """Half of the visual keys get a clearly larger logit; the cut falls inside the lower tie class."""
    nv, H, D, sys_len, text = 96, 2, 64, 1, 2
    cfg, ctx = _handmade(nv, H, D, sys_len, text, keep_bp=7500)
    try:
        g = torch.Generator().manual_seed(6)
        T0 = sys_len + nv + text
        K = torch.randn(1, 1, H, T0, D, generator=g)
        V = torch.randn(1, 1, H, T0, D, generator=g)
        q = torch.randn(1, 1, H, D, generator=g)
        lo, hi = K[:, :, :, sys_len:sys_len + 1].clone(), None
        hi = lo + 0.5 * q[:, :, :, None, :]                                          # larger q.k for every head
        strong = torch.zeros(nv, dtype=torch.bool)
        strong[torch.randperm(nv, generator=g)[:nv // 2]] = True
        K[:, :, :, sys_len:sys_len + nv] = torch.where(strong[None, None, None, :, None], hi, lo)
        out = torch.empty(1, 1, H, D, device="cuda")
        ctx.prefill_select(q.cuda(), K.cuda(), V.cuda(), [text], out)
        ids, cnt, _ = ctx.get_kept(0)
        n = int(cnt[0])
        assert n == 72
        weak_ids = [i for i in range(nv) if not strong[i]]
        want = set(i for i in range(nv) if strong[i]) | set(weak_ids[:72 - 48])      # all strong + lowest weak
        assert set(ids[0, :n].tolist()) == want
        assert ctx.status() == 0
    finally:
        ctx.close()


def test_inputs_from_a_producer_that_signals_completion_early():
    """q, k_new and v_new of every step are written by a kernel that allows its dependents to launch and only
    then, 30 us later, writes them.  In the default mode the step must still see the written values (its
    kernels start only when the producer's grid has finished): the outputs equal those of a run whose inputs
    were in place long before."""
    import native
    lib = native.load()
    wl = _small()
    a, b = GpuRun(wl), GpuRun(wl)
    try:
        a.prefill(); b.prefill()
        st = torch.cuda.current_stream().cuda_stream
        for t in range(1, 6):
            a.decode(t)
            q, kn, vn = b.inputs(t)
            src = torch.stack([q, kn, vn]).contiguous()
            dst = torch.zeros_like(src)                         # stale contents: zeros
            torch.cuda.synchronize()
            n16 = src.numel() * src.element_size() // 16
            assert lib.st3_test_early_trigger_copy(dst.data_ptr(), src.data_ptr(), n16, 30, st) == 0
            b.ctx.decode_step(t, dst[0], dst[1], dst[2], b.out)
            torch.cuda.synchronize()
            assert torch.equal(a.out, b.out), t
            for l in range(wl.num_layers):
                ia, ca, _ = a.kept(l)
                ib, cb, _ = b.kept(l)
                assert np.array_equal(ca, cb) and all(np.array_equal(ia[s, :ca[s]], ib[s, :cb[s]])
                                                      for s in range(wl.batch))
            b.check_rows_unit(0, 1, 0, t)                       # the appended rows are the written ones too
        assert a.ctx.status() == 0 and b.ctx.status() == 0
    finally:
        a.close(); b.close()


def test_a_new_generation_starts_at_layer_zero():
    """Prefilling layer 0 opens a new generation: layers that have not been prefilled again cannot decode."""
    wl = _small()
    run = GpuRun(wl)
    try:
        run.prefill()
        run.decode(1)
        g = run.g
        q0 = g.queries([0], device=run.dev)[0]
        K, V = g.prompt_kv([0, 1], device=run.dev)
        run.ctx.prefill_select(q0[0:2].contiguous(), K, V, g.text_len.tolist(), run.out[0:2], layer_begin=0)
        q, kn, vn = run.inputs(1)
        run.ctx.decode_step(1, q[0:2], kn[0:2], vn[0:2], run.out[0:2], layer_begin=0)     # prefilled again: fine
        with pytest.raises(B.St3Error) as e:                                              # layers 2.. are stale
            run.ctx.decode_step(1, q[2:], kn[2:], vn[2:], run.out[2:], layer_begin=2)
        assert e.value.code == 3
        with pytest.raises(B.St3Error) as e:
            run.ctx.decode_step(2, q[2:], kn[2:], vn[2:], run.out[2:], layer_begin=2)
        assert e.value.code == 3
        assert run.ctx.status() == 0
    finally:
        run.close()


@pytest.mark.parametrize("captured", [False, True])
def test_layer_calls_behind_a_copy_and_an_early_producer(captured):
    """Plain stream order, a call per layer: each layer's inputs are written by a kernel that allows its dependents to
    launch 20 us before it writes, the next layer's by a copy.  `captured`: the calls of a step are captured in a
    graph, which is launched once."""
    import native
    lib = native.load()
    wl = _small(num_layers=4)
    a, b = GpuRun(wl), GpuRun(wl)
    try:
        a.prefill(); b.prefill()
        for t in range(1, 4):
            a.decode(t)
            q, kn, vn = b.inputs(t)
            src = torch.stack([q, kn, vn], dim=1).contiguous()       # [layer][q | k | v]
            dst = torch.zeros_like(src)
            torch.cuda.synchronize()

            def step():
                st = torch.cuda.current_stream().cuda_stream
                for l in range(wl.num_layers):
                    if l % 2:
                        dst[l].copy_(src[l])
                    else:
                        n16 = src[l].numel() * src.element_size() // 16
                        assert lib.st3_test_early_trigger_copy(dst[l].data_ptr(), src[l].data_ptr(), n16, 20, st) == 0
                    b.ctx.decode_step(t, dst[l, 0:1], dst[l, 1:2], dst[l, 2:3], b.out[l:l + 1], layer_begin=l)

            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph):
                    step()
                graph.replay()
            else:
                step()
            torch.cuda.synchronize()
            assert torch.equal(a.out, b.out), t
            b.check_rows_unit(0, 1, 0, t)
        assert a.ctx.status() == 0 and b.ctx.status() == 0
    finally:
        a.close(); b.close()


def _score_sets(nv, g):
    """Scores that make the selection's histogram coarse, its bins full or the cut fall among equals."""
    u = torch.rand(nv, generator=g)
    wide = torch.exp((u - 0.5) * 160.0) * torch.where(torch.rand(nv, generator=g) < 0.5, -1.0, 1.0)
    tight = 1.0 + 1e-6 * u
    tight[nv // 3] = 3e38                                     # one outlier: everything else shares a bin
    steps = torch.floor(u * 7.0) - 3.0                        # seven levels, equal scores at the cut
    pairs = torch.floor(u * nv / 2.0)                         # a few keys to a bin, some of them equal
    n64 = torch.arange(nv, dtype=torch.float32) * 1e30        # 64 and 65 equal scores around the middle
    n65 = n64.clone()
    n64[nv // 2 - 32:nv // 2 + 32] = n64[nv // 2]
    n65[nv // 2 - 32:nv // 2 + 33] = n65[nv // 2]
    return dict(uniform=u, wide=wide, tight=tight, steps=steps, pairs=pairs, n64=n64, n65=n65, equal=torch.zeros(nv),
                tiny=u * 1e-42)


@pytest.mark.parametrize("nv,keep_bp", [(700, 5000), (700, 1), (2049, 3333), (8192, 5000), (65, 9999), (1, 5000), (300, 20), (513, 5000),
                                        (1025, 2000), (6401, 7777)])
def test_selection_over_hard_score_distributions(nv, keep_bp):
    cfg, ctx = _handmade(nv, H=1, keep_bp=keep_bp)
    try:
        g = torch.Generator().manual_seed(nv)
        T0 = 2 + nv + 3
        K, V = (torch.randn(1, 1, 1, T0, 64, generator=g) for _ in range(2))
        q, out = torch.randn(1, 1, 1, 64, generator=g).cuda(), torch.empty(1, 1, 1, 64, device="cuda")
        k = B.st3_schedule_count(cfg, 0, 0)
        for name, sc in _score_sets(nv, g).items():
            ctx.prefill_select_scored(q, K.cuda(), V.cuda(), [3], sc.float().view(1, 1, nv).cuda(), out)
            ids, cnt, _ = ctx.get_kept(0)
            order = np.lexsort((np.arange(nv), -sc.float().double().numpy()))
            assert int(cnt[0]) == k
            assert ids[0, :k].tolist() == sorted(order[:k].tolist()), name
            kv, vv, _, _ = ctx.get_rows(0, 0, 0)
            assert torch.equal(vv[:k].cpu(), V[0, 0, 0, 2 + ids[0, :k].long().cpu()]), name
        assert ctx.status() == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("H,nv", [(1, 17), (8, 256), (9, 257), (33, 511), (32, 513), (40, 576), (128, 700), (31, 1023),
                                  (32, 1028), (32, 1440), (32, 1460), (40, 2880)])
def test_selection_by_own_scores_at_the_edges_of_its_passes(H, nv):
    """Head counts and row counts around what a warp, a pass and the staged logits hold, rows on and off 16 bytes: the
    scores against 64 bits, the kept rows against an exact sort of those scores, and the rows moved with their ids."""
    D, sys_len, text, steps = 64, 2, 3, 4
    cfg, ctx = _handmade(nv, H, D, sys_len, text, steps=steps, keep_bp=9000)
    try:
        g = torch.Generator().manual_seed(1000 * H + nv)
        K, V = (torch.randn(1, 1, H, sys_len + nv + text, D, generator=g) for _ in range(2))
        q, kn, vn = (torch.randn(steps + 1, 1, 1, H, D, generator=g) for _ in range(3))
        out = torch.empty(1, 1, H, D, device="cuda")
        keys = K[0, 0].double()
        vis = list(range(nv))                                                       # rows held, in cache order
        for t in range(steps):
            if t == 0:
                ctx.prefill_select(q[0].cuda(), K.cuda(), V.cuda(), [text], out)
            else:
                ctx.decode_step(t, q[t].cuda(), kn[t].cuda(), vn[t].cuda(), out)
                keys = torch.cat([keys, kn[t, 0, 0].double()[:, None]], 1)
            rest = list(range(sys_len)) + list(range(sys_len + nv, keys.shape[1]))
            at = torch.tensor([sys_len + i for i in vis] + rest)
            p = torch.softmax(torch.einsum("hd,htd->ht", q[t, 0, 0].double(), keys[:, at]) / D ** 0.5, dim=1)
            want = p[:, :len(vis)].sum(0)
            ids, cnt, mass = ctx.get_kept(0)
            got = mass[0].cpu()[torch.tensor(vis)]
            assert torch.allclose(got.double(), want, rtol=5e-4, atol=0)            # fp32 dot products and ex2.approx
            k = B.st3_schedule_count(cfg, 0, t)
            best = np.array(vis)[np.lexsort((np.array(vis), -got.numpy()))[:k]]     # ties: the lower original index
            vis = ids[0, :k].tolist()
            assert int(cnt[0]) == k and 0 < k < nv and sorted(vis) == sorted(best.tolist())
            _, vv, _, _ = ctx.get_rows(0, 0, H - 1)
            assert torch.equal(vv[:k].cpu(), V[0, 0, H - 1, sys_len + torch.tensor(vis)])
        assert ctx.status() == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("H,nv", [(32, 729), (32, 2880), (24, 1152), (40, 2880), (16, 576)])
def test_ties_across_the_passes_over_the_staged_logits(H, nv):
    """Logits of a class are equal to the last bit by construction (keys with one entry); the rows of a class fall into
    several passes, the last of them short."""
    sys_len, text = 2, 3
    cfg, ctx = _handmade(nv, H, 64, sys_len, text, steps=8, keep_bp=9000)
    try:
        g = torch.Generator().manual_seed(nv + H)
        keys = torch.zeros(H, 15, 64)
        keys[:, :, 0] = torch.randn(H, 15, generator=g)
        _check_tied_classes(ctx, cfg, keys, torch.randn(4, 1, 1, H, 64, generator=g), "f32", sys_len, text, 15)
    finally:
        ctx.close()


def test_rows_off_16_bytes_are_selected_as_fast_as_rows_on_them():
    """Selection launches of a layer of eight sequences and 32 heads with 2877 and with 2880 visual tokens, in turn, the
    fastest generation of each: the copies of the logits are as wide for either (4-byte copies: 9 to 12 % slower)."""
    H, D, nb, steps = 32, 64, 8, 16
    runs, best = {}, {}
    try:
        for nv in (2877, 2880):
            ctx = B.Context(B.make_config(num_layers=1, num_heads=H, head_dim=D, dtype="bf16", batch=nb, sys_len=2, num_visual=nv,
                                          max_text_len=3, max_decode_steps=steps, stride=1, step_ratio_bp=0,
                                          first_prune_layer=0, first_ratio_bp=1000, tau=32.0))
            K, V = (torch.randn(1, nb, H, nv + 5, D, device="cuda").to(torch.bfloat16) for _ in range(2))
            runs[nv] = (ctx, K, V, torch.randn(steps + 1, 3, 1, nb, H, D, device="cuda").to(torch.bfloat16))
        out = torch.empty(1, nb, H, D, dtype=torch.bfloat16, device="cuda")
        for _ in range(8):
            for nv, (ctx, K, V, x) in runs.items():
                ctx.prefill_select(x[0, 0], K, V, [3] * nb, out)
                torch.cuda.synchronize()
                B.st3_profile_enable(ctx.handle, True)
                for t in range(1, steps + 1):
                    ctx.decode_step(t, x[t, 0], x[t, 1], x[t, 2], out)
                _, f_ms, _, n = B.st3_profile_read(ctx.handle)
                B.st3_profile_enable(ctx.handle, False)
                assert n == steps
                best[nv] = min(best.get(nv, 1e9), f_ms / n)
        assert best[2877] <= 1.04 * best[2880], best
    finally:
        for ctx, *_ in runs.values():
            ctx.close()


@pytest.mark.parametrize("nb,nv,H", [(50, 6400, 16), (38, 1536, 32), (3, 333, 5)])
def test_layers_of_a_stage_stay_alike_over_calls_of_different_sizes(nb, nv, H):
    """The pruning layer in a call of its own, the other layers of its stage in the next one, which may take selection
    blocks of another size: the same scores to the last bit, so the same tokens in the same order."""
    L, D, text, steps = 4, 64, 3, 3
    cfg = B.make_config(num_layers=L, num_heads=H, head_dim=D, dtype="bf16", batch=nb, sys_len=1, num_visual=nv,
                        max_text_len=text, max_decode_steps=steps, stride=L, step_ratio_bp=0, first_prune_layer=0,
                        first_ratio_bp=2000, tau=4.0, stage_shared=1)
    ctx = B.Context(cfg)
    try:
        g = torch.Generator(device="cuda").manual_seed(nv)
        rows = lambda *s: torch.empty(s, dtype=torch.bfloat16, device="cuda").normal_(generator=g)
        K, V = (rows(1, nb, H, 1 + nv + text, D).expand(L, -1, -1, -1, -1).contiguous() for _ in range(2))
        for t in range(steps + 1):
            q, kn, vn = (rows(L, nb, H, D) for _ in range(3))
            out = torch.empty_like(q)
            for l0, l1 in ((0, 1), (1, L)):
                if t == 0:
                    ctx.prefill_select(q[l0:l1], K[l0:l1], V[l0:l1], [text] * nb, out[l0:l1], layer_begin=l0)
                else:
                    ctx.decode_step(t, q[l0:l1], kn[l0:l1], vn[l0:l1], out[l0:l1], layer_begin=l0)
            n = B.st3_schedule_count(cfg, 0, t)
            ids, cnt, mass = ctx.get_kept(0)
            assert (cnt == n).all()
            for l in range(1, L):
                i, c, m = ctx.get_kept(l)
                assert torch.equal(c, cnt) and torch.equal(i[:, :n], ids[:, :n]) and torch.equal(m, mass), (t, l)
        assert ctx.status() == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("heads", [(40, 8), (8, 40)])
def test_contexts_of_different_sizes_used_in_turn(heads):
    """Their selections take different amounts of shared memory: neither context may take anything from the other."""
    nv, D, sys_len, text, steps = 576, 64, 2, 3, 3
    g = torch.Generator().manual_seed(9)
    data = {H: (torch.randn(steps + 1, 3, 1, 1, H, D, generator=g).cuda(),
                *(torch.randn(1, 1, H, sys_len + nv + text, D, generator=g).cuda() for _ in range(2))) for H in heads}

    def step(ctx, H, t):
        x, K, V = data[H]
        out = torch.empty(1, 1, H, D, device="cuda")
        if t == 0:
            ctx.prefill_select(x[0, 0], K, V, [text], out)
        else:
            ctx.decode_step(t, x[t, 0], x[t, 1], x[t, 2], out)
        return out

    alone = {}
    for H in heads:
        _, ctx = _handmade(nv, H, D, sys_len, text, steps=steps)
        alone[H] = [step(ctx, H, t) for t in range(steps + 1)]
        ctx.close()
    ctxs = {H: _handmade(nv, H, D, sys_len, text, steps=steps)[1] for H in heads}
    try:
        for t in range(steps + 1):
            for H in heads:
                assert torch.equal(step(ctxs[H], H, t), alone[H][t]), (H, t)
        assert all(c.status() == 0 for c in ctxs.values())
    finally:
        for c in ctxs.values():
            c.close()


def test_more_heads_sequences_and_layers_than_a_grid_dimension_holds():
    """65 536 (layer, sequence, head) units in one call: 64 sequences of the same contents against one of them."""
    L, H, D, nv, text, nb = 32, 32, 64, 8, 3, 64
    T0 = 1 + nv + text
    g = torch.Generator().manual_seed(12)
    rows = lambda *s: torch.randn(*s, generator=g).to(torch.bfloat16).cuda()
    q, K, V = rows(L, 1, H, D), rows(L, 1, H, T0, D), rows(L, 1, H, T0, D)
    q1, k1, v1 = rows(L, 1, H, D), rows(L, 1, H, D), rows(L, 1, H, D)
    res = []
    for n in (1, nb):
        cfg = B.make_config(num_layers=L, num_heads=H, head_dim=D, dtype="bf16", batch=n, sys_len=1, num_visual=nv,
                            max_text_len=text, max_decode_steps=1, stride=7, step_ratio_bp=1000, tau=4.0)
        ctx = B.Context(cfg)
        try:
            many = lambda t: t.expand(t.shape[0], n, *t.shape[2:]).contiguous()
            out0, out1 = torch.empty_like(many(q)), torch.empty_like(many(q))
            ctx.prefill_select(many(q), many(K), many(V), [text] * n, out0)
            kept = [ctx.get_kept(l)[:2] for l in range(L)]
            ctx.decode_step(1, many(q1), many(k1), many(v1), out1)
            assert ctx.status() == 0
            res.append((out0, out1, kept))
        finally:
            ctx.close()
    (a0, a1, ka), (b0, b1, kb) = res
    assert torch.equal(a0.expand_as(b0), b0) and torch.equal(a1.expand_as(b1), b1)
    for (ia, ca), (ib, cb) in zip(ka, kb):
        c = int(ca[0])
        assert (cb == c).all() and torch.equal(ia[:, :c].expand(nb, c), ib[:, :c])


def _check_selection_launches(nb, nv, H, kernel):
    """A prompt and two steps of `nb` sequences in one layer, through the named form of the selection kernel only: outputs
    and scores against 64 bits, the kept rows against an exact sort of the scores, and the rows moved with their ids."""
    D, sys_len, text, steps = 64, 1, 2, 2
    cfg = B.make_config(num_layers=1, num_heads=H, head_dim=D, dtype="bf16", batch=nb, sys_len=sys_len, num_visual=nv,
                        max_text_len=text, max_decode_steps=steps, stride=1, step_ratio_bp=0, first_prune_layer=0, tau=8.0)
    ctx = B.Context(cfg)
    try:
        g = torch.Generator(device="cuda").manual_seed(nv)
        rows = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
        K, V = rows(nb, H, sys_len + nv + text, D), rows(nb, H, sys_len + nv + text, D)
        q, kn, vn = (rows(steps + 1, 1, nb, H, D) for _ in range(3))
        out = torch.empty_like(q)
        held = torch.ones(nb, nv, dtype=torch.bool, device="cuda")
        keys, vals = K, V
        for t in range(steps + 1):
            with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA], acc_events=True) as prof:
                if t == 0:
                    ctx.prefill_select(q[0], K[None], V[None], [text] * nb, out[0])
                else:
                    ctx.decode_step(t, q[t], kn[t], vn[t], out[t])
                torch.cuda.synchronize()
            names = [e.key for e in prof.key_averages() if "st3_finish_kernel" in e.key]
            assert len(names) == 1 and kernel in names[0], names
            if t:
                keys, vals = (torch.cat([x, n[t, 0][:, :, None]], 2) for x, n in ((keys, kn), (vals, vn)))
            gone = torch.zeros(nb, keys.shape[2], dtype=torch.bool, device="cuda")
            gone[:, sys_len:sys_len + nv] = ~held
            x = torch.einsum("bhd,bhtd->bht", q[t, 0].double(), keys.double()) / D ** 0.5
            p = torch.softmax(x.masked_fill(gone[:, None], float("-inf")), dim=2)
            ref = torch.einsum("bht,bhtd->bhd", p, vals.double())
            assert (out[t, 0].double() - ref).abs().max() <= 2e-2 * ref.abs().max()
            ids, cnt, mass = ctx.get_kept(0)
            want = p[:, :, sys_len:sys_len + nv].sum(1)
            assert torch.allclose(mass[held].double(), want[held], rtol=5e-4, atol=0)   # fp32 dot products and ex2.approx
            n = B.st3_schedule_count(cfg, 0, t)
            best = mass.masked_fill(~held, -1.0).sort(dim=1, descending=True, stable=True).indices[:, :n]
            assert (cnt == n).all() and torch.equal(ids[:, :n].sort(dim=1).values, best.sort(dim=1).values.int())
            held = torch.zeros_like(held).scatter_(1, best, True)
        for b, h in ((0, 0), (nb - 1, H - 1)):
            kv, vv, _, _ = ctx.get_rows(0, b, h)
            at = sys_len + ids[b, :n].long()
            assert torch.equal(kv[:n], K[b, h, at]) and torch.equal(vv[:n], V[b, h, at])
        assert ctx.status() == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("nv,H,kernel", [(6399, 3, "64, 2, 512>"), (6400, 3, "64, 1, 1024>"), (700, 33, "64, 2, 512>")])
def test_half_size_selection_blocks_up_to_what_two_of_them_leave_of_an_sm(nv, H, kernel):
    """More units than SMs: two selection blocks of 512 threads to an SM, as long as their shared memory fits twice."""
    _check_selection_launches(150, nv, H, kernel)


@pytest.mark.parametrize("nb,nv,H,kernel", [(74, 300, 33, "64, 1, 512>"), (75, 300, 33, "64, 1, 1024>"),
                                            (111, 577, 32, "64, 1, 1024>"), (112, 577, 32, "64, 2, 512>"),
                                            (112, 1500, 32, "64, 1, 1024>"), (148, 300, 17, "64, 2, 512>")])
def test_selection_blocks_of_a_crowded_launch(nb, nv, H, kernel):
    """From half as many units as SMs, blocks of 1024 threads; from three quarters, two blocks to an SM if they hold all rows
    at a time (148 SMs)."""
    _check_selection_launches(nb, nv, H, kernel)


def test_profile_counts_the_copy_of_a_prompts_kept_rows():
    """The select/compact time of a prompt holds the copy of the kept rows: it is no shorter than their bytes take at
    8 TB/s, less what the L2 cache (126 MB) may still hold of either side.  The selection alone is far shorter."""
    L, H, nb, D, nv = 3, 32, 8, 128, 2880
    cfg = B.make_config(num_layers=L, num_heads=H, head_dim=D, dtype="bf16", batch=nb, sys_len=4, num_visual=nv,
                        max_text_len=4, max_decode_steps=1, stride=3, step_ratio_bp=0, first_prune_layer=0, tau=4.0)
    ctx = B.Context(cfg)
    try:
        q = torch.randn(L, nb, H, D, device="cuda").to(torch.bfloat16)
        K, V = (torch.randn(L, nb, H, nv + 8, D, device="cuda", dtype=torch.bfloat16) for _ in range(2))
        out = torch.empty_like(q)
        B.st3_profile_enable(ctx.handle, True)
        for _ in range(3):
            ctx.prefill_select(q, K, V, [4] * nb, out)
        _, f_ms, _, nf = B.st3_profile_read(ctx.handle)
        moved = 2 * 2 * L * nb * H * (nv // 2) * D * 2            # K and V, read and written
        assert nf == 3 and f_ms / nf * 1e-3 >= (moved - 2 * 126e6) / 8e12, f_ms / nf
        assert ctx.status() == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("lazy", [False, True])
def test_a_wait_that_runs_out_is_reported(lazy):
    """A flag that nothing sets: the attention launch gives up after its limit, waits for its copies in flight and ends;
    the host reads the status, and a context of its own works as before."""
    kw = dict(stage_shared=1, lazy_mask=0b101010) if lazy else {}
    wl = _small(first_prune_layer=2, stride=4)
    run, after = GpuRun(wl, **kw), GpuRun(wl, **kw)
    try:
        run.prefill()
        run.decode(1)
        words = run.ctx.workspace[run.ctx._ws_ptr - run.ctx.workspace.data_ptr():][:run.ctx.workspace_bytes // 256 * 256]
        words = words.view(torch.int32).view(-1, 64)
        n = wl.num_layers * wl.batch                            # one flag per (layer, sequence), 256-byte aligned
        before = (words[:, :n] == 2).all(1)                     # the second call of the context
        run.decode(2)
        where = (before & (words[:, :n] == 3).all(1)).nonzero().flatten()
        assert where.numel() == 1
        words[where[0], :n] = -1000
        torch.cuda.synchronize()
        run.decode(3)
        assert run.ctx.status(raise_on_error=False) & B.DEV_COPY_TIMEOUT
        after.prefill()
        for t in range(1, 4):
            before_step = after.snapshot(range(wl.num_layers))
            after.decode(t)
        for l in range(wl.num_layers):
            after.check_decode_unit(0, l, 3, before_step[l])
        assert after.ctx.status() == 0
    finally:
        run.close(); after.close()
