"""GPU tests of the steps around the tasks: the task table and the task order of a built model, the pruning step and
the cost estimate against measured times, one latency-gated iteration of the pruning loop, and the bounded waits."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cp():
    import paper_2207_01260_b200 as m
    m.lib()
    return m


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _small_resnet(batch=8, hw=64):
    from paper_2207_01260_b200.pipeline import PrunedNetwork
    table = wl.resnet18()
    table["input"] = (hw, hw, 3)
    weights = wl.model_weights(table)
    return table, weights, PrunedNetwork(table, weights, batch), wl.model_input(table, batch)


def test_a_bounded_wait_that_expires_reports_a_timeout_and_leaves_the_device_usable(cp):
    cp.cprune_poll_device_status()
    cp.cprune_selftest_wait_timeout()
    with pytest.raises(cp.CpruneError) as e:
        cp.cprune_poll_device_status()
    assert e.value.status == 5                    # CPRUNE_ERR_TIMEOUT
    cp.cprune_poll_device_status()                # the word was cleared: OK again
    # a normal task still runs and is right
    x, w, b, _ = wl.conv_task_tensors(3, 2, 64, 14, 14, 48, 3, 3)
    plan = cp.cprune_task_plan(2, 64, 14, 14, 48, 3, 3, 1, 1)
    wp, bp = cp.cprune_pack_weights(plan, _dev(w), _dev(b))
    y = cp.cprune_task_run(plan, cp.cprune_cast_input(_dev(x)), wp, bp).float().cpu().numpy()
    cp.cprune_poll_device_status()
    ref, bound = oracle.conv2d(x, w, b, 1, 1, 1, "relu", with_bound=True)
    assert np.max(np.abs(y[..., :48] - ref) / bound) <= 2e-2


def test_task_table_times_and_order_of_a_model(cp):
    table, weights, net, x = _small_resnet()
    net.run(_dev(x))
    entries = net.model.task_table()
    # the oracle's grouping of the same table: same number of distinct tasks, same multiplicities, same first members
    ref = oracle.task_table(table)
    assert len(entries) == len(ref) == 15 and sum(c for _, c, _ in entries) == 20
    assert [c for _, c, _ in entries] == [len(names) for _, names in ref]
    ms = net.model.time_tasks(reps=4)
    cp.cprune_poll_device_status()
    assert len(ms) == 15 and all(0 < t < 50 for t in ms)
    pri = net.task_priorities(reps=4)
    assert sorted(sum((p["layers"] for p in pri), [])) == sorted(n for _, names in ref for n in names)
    impacts = [p["impact"] for p in pri]
    assert impacts == sorted(impacts, reverse=True)
    assert [p["count"] for p in pri] == [len(p["layers"]) for p in pri]
    # the library's order of these very measurements is the oracle's
    t, c = [p["ms"] for p in pri], [p["count"] for p in pri]
    assert cp.cprune_task_order(t, c) == oracle.task_order(t, c)


def test_times_of_tasks_that_run_as_one_kernel(cp):
    # 288 -> 64 channels, 14x14, 64 images: one kernel takes about two thirds of what the two take (13.0 and 8.9 us in a network); launches
    # one by one begin on a grid of about 2.06 us, by which either time may be off
    N, C, H, K = 64, 288, 14, 64
    dw, pj = cp.cprune_task_plan(N, C, H, H, C, 3, 3, 1, 1, C), cp.cprune_task_plan(N, C, H, H, K, 1, 1, 1, 0)
    g = torch.Generator(device="cuda").manual_seed(5)
    rand = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    p1, p2 = cp.cprune_pack_weights(dw, rand(C, 1, 3, 3), rand(C)), cp.cprune_pack_weights(pj, rand(K, C, 1, 1), rand(K))
    fc = cp.cprune_fc_pack(rand(8, K))

    def build(flags):
        # a chain of two blocks with the same plans: 0 -> dw -> 1 -> 1x1 -> 2 -> expand -> 3 -> dw -> 4 -> 1x1 -> 5
        ex = cp.cprune_task_plan(N, K, H, H, C, 1, 1, 1, 0)
        p3 = cp.cprune_pack_weights(ex, rand(C, K, 1, 1), rand(C))
        conv = lambda i, plan, p, f=0: cp.TaskDesc(op=cp.OP_CONV, in_=i, out=i + 1, res=-1, plan=plan.handle, w=p[0].data_ptr(), b=p[1].data_ptr(), p0=f)
        tasks = [conv(0, dw, p1, flags[0]), conv(1, pj, p2), conv(2, ex, p3), conv(3, dw, p1, flags[1]), conv(4, pj, p2),
                 cp.TaskDesc(op=cp.OP_GAP, in_=5, out=6, res=-1), cp.TaskDesc(op=cp.OP_FC, in_=6, out=7, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=K, p1=8)]
        return cp.cprune_model_create(N, H, H, C, tasks, keep_alive=(dw, pj, ex, p1, p2, p3, fc))

    one = cp.CONV_WITH_NEXT
    times = {}
    for flags in ((0, 0), (one, one), (one, 0)):
        model = build(flags)
        assert [c for _, c, _ in model.task_table()] == [2, 2, 1]
        runs = [model.time_tasks(reps=20) for _ in range(3)]
        times[flags] = min(t[0] + t[1] for t in runs)
        assert all(0 < v < 1 for t in runs for v in t)
    cp.cprune_poll_device_status()
    print("\ndepthwise + 1x1, ms: separate %.4f, one kernel %.4f, one of two blocks as one kernel %.4f" % tuple(times.values()))
    # measured ratio 0.6 to 0.7: 0.85 is above it by more than a step of the grid (2.06 of about 14 us)
    assert times[(one, one)] < 0.85 * times[(0, 0)]
    assert times[(one, one)] < times[(one, 0)] < times[(0, 0)]


def test_one_latency_gated_iteration_of_the_pruning_loop(cp):
    from paper_2207_01260_b200 import search
    from paper_2207_01260_b200.pipeline import PrunedNetwork
    table, weights, net, x = _small_resnet()
    xd = _dev(x)
    # a target no candidate can miss, so that the first prunable task in priority order is accepted
    out = search.latency_gated_iteration(table, weights, 8, xd, target_ms=1e9)
    assert out["accepted"] and out["ms"] < out["target_ms"]
    rec = out["tried"][-1]
    by = wl.layer_by_name(out["table"])
    old = wl.layer_by_name(table)
    for name in rec["pruned"]:
        assert by[name]["keep"] == old[name]["keep"] - rec["step"] and rec["step"] >= 8
    assert all(by[n]["keep"] == old[n]["keep"] for n in by if by[n]["kind"] == "conv" and n not in rec["pruned"])
    # tasks tried before it had no prunable layer (block outputs and shortcut convs keep their width in this table)
    for r in out["tried"][:-1]:
        assert r["candidate_ms"] is None
    # the accepted candidate is a correct network: logits against the oracle on the candidate table
    logits = out["net"].run(xd).cpu().numpy()
    cp.cprune_poll_device_status()
    pw, _ = oracle.prune_model(out["table"], weights)
    ref = oracle.model_ref(out["table"], pw, x, matched=True)
    assert np.linalg.norm(logits - ref) <= 1e-2 * np.linalg.norm(ref)
    # a target no candidate can reach: every task is tried, none accepted, the model stays as it was
    out2 = search.latency_gated_iteration(table, weights, 8, xd, target_ms=0.0)
    assert not out2["accepted"] and out2["table"] is table and len(out2["tried"]) == 15


def _time_task(cp, plan, x, wp, bp, reps=20):
    # The runs are replayed as a CUDA graph.  Launched one by one they begin on a grid of about 2.06 us: a task then takes 18.6 or 20.6 us
    # (a ratio of 0.902, whatever the kernel does in between), and the bounds below could not be told from a step of that clock.
    # In graphs the levels of the three shapes are flat to 4 % (the bound is 15 %), and the cheapest is 0.86, 0.66 and 0.54 of the dearest
    # (the bound is 0.9).
    y = torch.empty((plan.N, plan.out_h, plan.out_w, plan.k_pad), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(max(plan.workspace_bytes, 16), dtype=torch.uint8, device="cuda")
    for _ in range(3):
        cp.cprune_task_run(plan, x, wp, bp, None, y, ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(reps):
            cp.cprune_task_run(plan, x, wp, bp, None, y, ws)
    graph.replay()
    best = 1e9
    for _ in range(3):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        graph.replay()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) / reps)
    return best


@pytest.mark.parametrize("shape", [(64, 128, 28, 28, 128, 3, 1, 1), (64, 64, 56, 56, 64, 3, 1, 1), (64, 256, 14, 14, 256, 3, 1, 1)])
def test_estimated_steps_against_measured_levels(cp, shape):
    # Within one level of the estimate (filter counts the cost model prices the same) the measured time is flat; across
    # the whole sweep the cheapest estimated level is measurably faster than the dearest.  (The paper's point, Sec. 3.5:
    # time falls in steps, so pruning fewer filters than a step buys nothing.)
    N, C, H, W, K, R, stride, pad = shape
    full = cp.cprune_task_plan(N, C, H, W, K, R, R, stride, pad)
    step = cp.cprune_prune_step(full)
    assert step in (16, 32, 64, 128)
    x = torch.randn((N, H, W, full.c_pad), device="cuda").to(torch.bfloat16)
    w = torch.randn((K, C, R, R), device="cuda") * 0.05
    levels = {}
    for k in range(K, K // 4 - 1, -3):
        plan = cp.cprune_task_plan(N, C, H, W, k, R, R, stride, pad)
        wp, bp = cp.cprune_pack_weights(plan, w[:k].contiguous(), torch.zeros(k, device="cuda"))
        est = cp.cprune_task_estimate(full, k)
        assert est == pytest.approx(plan.est_us)
        levels.setdefault(round(est, 4), []).append(_time_task(cp, plan, x, wp, bp))
    cp.cprune_poll_device_status()
    assert len(levels) >= 3
    for est, ts in levels.items():
        assert max(ts) <= 1.15 * min(ts), ("a level of the estimate is not flat in the measurement", est, ts)
    keys = sorted(levels)
    assert np.median(levels[keys[0]]) < 0.9 * np.median(levels[keys[-1]]), {k: np.median(v) for k, v in levels.items()}
    # no filter count inside the full-width level is cheaper than full width by more than noise: pruning less than a
    # step does not pay
    print("\n%s: step %d; levels (est us -> measured ms): %s" % (shape, step, {k: round(float(np.median(v)), 4) for k, v in levels.items()}))
