"""Parity of the CUDA library (through its C ABI) against the CPU oracle, element by element."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

TOL = 2e-2          # the contract: max |err| <= TOL * (|b| + sum |x||w| + |res|) per output element, against the exact oracle
# The engineering bound, against the matched oracle (x, w and the residual rounded to bfloat16, float64 arithmetic): what
# is left is the rounding of the stored result to bfloat16 (half a unit in the 8th significant bit: 2^-8 |ref|, taken
# twice here) and the float32 accumulation on the device (a few 1e-6 of the scale; 1e-4 allows for worst-case orders).
# A dropped channel block, tap or tile-edge column changes an output by about 1e-2 of the scale and fails this check.
MATCH_REL, MATCH_ABS = 2.0 ** -7, 1e-4
WORST = {}          # test name -> (worst contract ratio, worst matched ratio), printed at the end of the session


def check_values(name, got, exact, bound, matched, bound_m):
    """got vs the exact oracle under the contract and vs the matched oracle under the engineering bound."""
    r1 = float(np.max(np.abs(got - exact) / (bound + 1e-30)))
    r2 = float(np.max(np.abs(got - matched) / (MATCH_REL * np.abs(matched) + MATCH_ABS * bound_m + 1e-30)))
    prev = WORST.get(name, (0.0, 0.0))
    WORST[name] = (max(prev[0], r1), max(prev[1], r2))
    assert r1 <= TOL, (name, "contract", r1)
    assert r2 <= 1.0, (name, "matched", r2, np.unravel_index(np.argmax(np.abs(got - matched) - MATCH_REL * np.abs(matched) - MATCH_ABS * bound_m), got.shape))
    return r1, r2


@pytest.fixture(scope="module", autouse=True)
def _report_worst_ratios():
    yield
    if WORST:
        print("\nworst error ratios (contract: err / (2e-2-scale bound) must be <= 2e-2; matched: must be <= 1):")
        for k in sorted(WORST):
            print("  %-58s contract %.2e   matched %.3f" % (k, WORST[k][0], WORST[k][1]))


@pytest.fixture(scope="module")
def cp():
    import paper_2207_01260_b200 as m
    m.lib()
    return m


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def run_task(cp, x, w, b, stride, pad, groups=1, act="relu", res=None, pool=None, kernel="auto", flags=()):
    N, H, W, C = x.shape
    K, _, R, S = w.shape
    plan = cp.cprune_task_plan(N, C, H, W, K, R, S, stride, pad, groups, act, res is not None, pool, kernel, flags)
    xb = cp.cprune_cast_input(_dev(x))
    wp, bp = cp.cprune_pack_weights(plan, _dev(w), _dev(b))
    rb = cp.cprune_cast_input(_dev(res)) if res is not None else None
    y = cp.cprune_task_run(plan, xb, wp, bp, rb)
    cp.cprune_poll_device_status()
    return y.float().cpu().numpy(), plan


def _pooled(ref, bound, pool):
    # the error bound of a maximum is at most the largest bound in its window
    if pool == "max3x3s2":
        return oracle.maxpool(ref, 3, 2, 1), oracle.maxpool(bound, 3, 2, 1)
    if pool:
        return oracle.maxpool(ref, 2, 2, 0), oracle.maxpool(bound, 2, 2, 0)
    return ref, bound


def check_task(cp, N, C, H, W, K, R, stride, pad, groups=1, act="relu", with_res=False, pool=None, kernel="auto",
               seed=11, flags=(), name=None):
    P, Q = oracle.out_size(H, R, stride, pad), oracle.out_size(W, R, stride, pad)
    x, w, b, res = wl.conv_task_tensors(seed, N, C, H, W, K, R, R, groups, with_res, P, Q)
    y, plan = run_task(cp, x, w, b, stride, pad, groups, act, res, pool, kernel, flags)
    ref, bound = _pooled(*oracle.conv2d(x, w, b, stride, pad, groups, act, res, with_bound=True), pool)
    rb = oracle.round_bf16
    ref_m, bound_m = _pooled(*oracle.conv2d(rb(x), rb(w), b, stride, pad, groups, act, None if res is None else rb(res),
                                            with_bound=True), pool)
    assert y.shape == (N, plan.out_h, plan.out_w, plan.k_pad)
    assert np.all(y[..., K:] == 0), "pad lanes must be written as zero"
    label = name or "task N%d C%d %dx%d K%d R%d s%d g%d %s%s%s %s" % (N, C, H, W, K, R, stride, groups, act, "+res" if with_res else "",
                                                                       "+" + pool if pool else "", kernel)
    check_values(label, y[..., :K], ref, bound, ref_m, bound_m)
    assert np.max(np.abs(y[..., :K] - ref)) > 0 or np.max(np.abs(ref)) == 0   # bf16 data cannot be bit-exact against float64
    return plan


# ------------------------------------------------------------------ selection (bit-exact)

@pytest.mark.parametrize("K,C,R,keep", [(64, 64, 3, 48), (37, 5, 3, 17), (512, 512, 3, 358), (96, 16, 1, 72),
                                        (1280, 7, 1, 999), (9, 3, 7, 1), (300, 20, 3, 300)])
def test_select_filters_bit_exact(cp, K, C, R, keep):
    w = wl.normal_f32(21, 1, (K, C, R, R), 0.05)
    if K >= 30:
        w[11] = w[3]
        w[20] = -w[3]
    b = wl.normal_f32(21, 2, (K,), 0.01)
    wn = wl.normal_f32(21, 3, (13, K, 3, 3), 0.05)
    kept, wo, bo, wno = cp.cprune_select_filters(_dev(w), keep, _dev(b), _dev(wn))
    cp.cprune_poll_device_status()
    rk, rw, rb, rwn = oracle.select_filters(w, b, keep, wn)
    assert np.array_equal(kept.cpu().numpy(), rk)
    assert wo.cpu().numpy().tobytes() == rw.tobytes()
    assert bo.cpu().numpy().tobytes() == rb.tobytes()
    assert wno.cpu().numpy().tobytes() == rwn.tobytes()
    wd = wl.normal_f32(21, 4, (K, 1, 3, 3), 0.05)
    kept2, _, _, wdo = cp.cprune_select_filters(_dev(w), keep, None, _dev(wd), next_is_depthwise=True)
    assert np.array_equal(kept2.cpu().numpy(), rk)
    assert wdo.cpu().numpy().tobytes() == wd[rk].tobytes()
    g = cp.cprune_gather_columns(_dev(wn), kept)
    assert g.cpu().numpy().tobytes() == rwn.tobytes()
    g = cp.cprune_gather_rows(_dev(b), kept)
    assert g.cpu().numpy().tobytes() == rb.tobytes()


@pytest.mark.parametrize("K,C,R,keep,nxt", [(1, 1, 1, 1, (3, 1)), (257, 3, 3, 255, (2, 3)), (1280, 30, 1, 700, (900, 1)), (8192, 2, 1, 4000, (1, 5)),
                                            (8200, 1, 1, 7000, (2, 1)), (300, 64, 3, 150, None)])
def test_select_and_slice_edges(cp, K, C, R, keep, nxt):
    # radix selection with exact ties and equal norms everywhere, rows copied as vectors and as single elements, several blocks
    # per consumer row, a depthwise consumer (None), and more filters than the one-kernel path holds (8200)
    w = wl.normal_f32(93, 1, (K, C, R, R), 0.05)
    w[: K // 2] = w[K // 3]                                     # half of the filters tie exactly
    b = wl.normal_f32(93, 2, (K,), 0.01)
    wn = wl.normal_f32(93, 3, (K, 1, 3, 3) if nxt is None else (nxt[0], K, nxt[1], nxt[1]), 0.05)
    kept, wo, bo, wno = cp.cprune_select_filters(_dev(w), keep, _dev(b), _dev(wn), nxt is None)
    cp.cprune_poll_device_status()
    idx = oracle.select_indices(w, keep)
    assert np.array_equal(kept.cpu().numpy(), idx)
    assert np.array_equal(wo.cpu().numpy(), w[idx]) and np.array_equal(bo.cpu().numpy(), b[idx])
    assert np.array_equal(wno.cpu().numpy(), wn[idx] if nxt is None else wn[:, idx])


def test_select_every_keep_count_nests(cp):
    w = wl.normal_f32(22, 1, (64, 64, 3, 3), 0.06)
    dw = _dev(w)
    for keep in range(16, 65):
        kept, _, _, _ = cp.cprune_select_filters(dw, keep)
        assert np.array_equal(kept.cpu().numpy(), oracle.select_indices(w, keep))


def test_select_flags_bad_weights_and_bad_arguments(cp):
    w = wl.normal_f32(23, 1, (8, 4, 3, 3), 0.05)
    w[2, 1, 1, 1] = np.nan
    cp.cprune_select_filters(_dev(w), 4)
    with pytest.raises(cp.CpruneError) as e:
        cp.cprune_poll_device_status()
    assert e.value.status == 7
    cp.cprune_poll_device_status()      # the word was cleared
    good = _dev(wl.normal_f32(23, 2, (8, 4, 3, 3), 0.05))
    for keep in (0, 9, -1):
        with pytest.raises(cp.CpruneError) as e:
            cp.cprune_select_filters(good, keep)
        assert e.value.status == 1
    with pytest.raises(cp.CpruneError) as e:
        cp.cprune_select_filters(good, 4, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    assert e.value.status == 3


@pytest.mark.parametrize("K", [64, 300, 8200])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_filters_that_hold_no_numbers_rank_last(cp, K, value):
    # the data breaks the precondition (and the status word says so), but the order is that of signed norms on both paths: the
    # integer sums of these filters are negative
    w = wl.normal_f32(26, 1, (K, 4, 3, 3), 0.05)
    bad = [7, K // 2, K - 1]
    for k in bad:
        w[k, 1, 1, 1] = value
    zeroed = w.copy()
    zeroed[bad] = 0
    for keep in (1, K // 3, K - len(bad)):
        kept = cp.cprune_select_filters(_dev(w), keep)[0].cpu().numpy()
        shared = cp.cprune_select_shared([_dev(w)], keep).cpu().numpy()
        with pytest.raises(cp.CpruneError) as e:
            cp.cprune_poll_device_status()
        assert e.value.status == 7
        assert np.array_equal(kept, oracle.select_indices(zeroed, keep)) and np.array_equal(shared, kept)


# ------------------------------------------------------------------ single tasks

def test_config1_single_pruned_task(cp):
    m = wl.single_task()
    w, b = wl.model_weights(m)["conv"]
    x = wl.model_input(m, 1)
    kept, wo, bo, _ = cp.cprune_select_filters(_dev(w), 48, _dev(b))
    rk, rw, rb, _ = oracle.select_filters(w, b, 48)
    assert np.array_equal(kept.cpu().numpy(), rk)
    for kernel in ("tensor", "direct"):
        y, plan = run_task(cp, x, wo.cpu().numpy(), bo.cpu().numpy(), 1, 1, kernel=kernel)
        assert cp.KERNEL_NAMES[plan.kernel] == kernel
        ref, bound = oracle.conv2d(x, rw, rb, 1, 1, 1, "relu", with_bound=True)
        ref_m, bound_m = oracle.conv2d(oracle.round_bf16(x), oracle.round_bf16(rw), rb, 1, 1, 1, "relu", with_bound=True)
        assert y.shape == (1, 32, 32, 48)
        check_values("config 1 (%s)" % kernel, y, ref, bound, ref_m, bound_m)


DENSE_CASES = [
    # N, C, H, W, K, R, stride, pad
    (1, 64, 32, 32, 48, 3, 1, 1),
    (2, 44, 13, 17, 101, 3, 1, 1),
    (3, 8, 9, 9, 16, 3, 1, 1),
    (1, 24, 20, 20, 45, 1, 1, 0),
    (2, 72, 14, 14, 24, 1, 1, 0),
    (1, 100, 15, 11, 130, 3, 2, 1),
    (2, 130, 9, 10, 260, 3, 1, 1),
    (1, 64, 28, 28, 128, 1, 2, 0),
    (2, 16, 12, 12, 300, 3, 1, 0),
    (1, 40, 23, 23, 58, 7, 2, 3),
    (5, 187, 8, 8, 171, 3, 1, 1),
    (3, 212, 2, 2, 198, 3, 1, 1),
    (1, 320, 7, 7, 1280, 1, 1, 0),
]


@pytest.mark.parametrize("kernel", ["tensor", "direct"])
@pytest.mark.parametrize("case", DENSE_CASES)
def test_dense_task_parity(cp, case, kernel):
    N, C, H, W, K, R, stride, pad = case
    plan = check_task(cp, N, C, H, W, K, R, stride, pad, kernel=kernel)
    assert cp.KERNEL_NAMES[plan.kernel] == kernel


@pytest.mark.parametrize("kernel", ["tensor", "direct"])
def test_dense_task_epilogues(cp, kernel):
    check_task(cp, 2, 44, 14, 14, 64, 3, 1, 1, act="relu", with_res=True, kernel=kernel)
    check_task(cp, 1, 72, 14, 14, 24, 1, 1, 0, act="none", with_res=True, kernel=kernel)
    check_task(cp, 2, 24, 16, 16, 108, 1, 1, 0, act="relu6", kernel=kernel)
    check_task(cp, 2, 45, 16, 16, 58, 3, 1, 1, act="relu", pool="max2x2", kernel=kernel)
    check_task(cp, 1, 64, 8, 8, 64, 3, 1, 1, act="none", kernel=kernel)


@pytest.mark.parametrize("case", [
    # N, C, HW, K: fused in the filter-major epilogue (Q = 32, 16, 4), in the pixel-major epilogue (Q = 8, 2),
    # in the split-K finalize kernel (few tiles), and as a separate pass (Q not a power of two)
    (3, 45, 32, 58), (2, 101, 16, 96), (5, 20, 4, 40), (4, 171, 8, 163), (40, 64, 2, 243), (2, 250, 4, 212),
    (1, 24, 12, 32), (1, 200, 12, 200)])
def test_fused_maxpool(cp, case):
    N, C, HW, K = case
    check_task(cp, N, C, HW, HW, K, 3, 1, 1, act="relu", pool="max2x2", kernel="tensor")


def test_pointwise_tasks_as_flat_matrix_products(cp):
    # 1x1 stride-1 tasks with enough pixels run on the patch kernel with all pixels viewed as one row: ragged last tile,
    # residual through the staging buffer, several filter tiles, channel counts off the 16 / 64 grid
    plan = check_task(cp, 8, 24, 56, 56, 108, 1, 1, 0, act="relu6", kernel="tensor")
    assert plan.variant == 1
    check_task(cp, 3, 108, 57, 59, 24, 1, 1, 0, act="none", with_res=True, kernel="tensor")
    check_task(cp, 5, 72, 40, 41, 300, 1, 1, 0, act="relu", kernel="tensor")
    check_task(cp, 64, 320, 7, 7, 1280, 1, 1, 0, act="relu6", kernel="tensor")
    # one filter tile: the tile is staged pixel by pixel as it lies in memory (variant 2).  A pixel pitch of an odd number of
    # 16-byte pieces (or 32 bytes) leaves by one bulk copy (one and two 64-filter groups, with and without residual, ragged
    # last tile); an even number is staged one piece longer and leaves by one tiled copy whose box is wider than the tensor
    # (without residual; with one such tasks keep the 64-filter-wide stores of variant 1)
    for case in ((12, 16, 50, 53, 72, "relu6", False, 2), (6, 32, 47, 50, 16, "none", False, 2), (4, 150, 45, 46, 40, "relu6", True, 2),
                 (8, 48, 45, 46, 88, "relu", True, 2), (8, 48, 45, 46, 133, "relu", False, 2), (5, 24, 44, 45, 64, "relu", False, 2),
                 (7, 40, 33, 35, 32, "relu6", False, 2), (8, 48, 45, 46, 133, "relu", True, 1), (5, 24, 44, 45, 64, "none", True, 1)):
        N, C, H, W, K, act, res, variant = case
        plan = check_task(cp, N, C, H, W, K, 1, 1, 0, act=act, with_res=res, kernel="tensor")
        assert plan.variant == variant, case


@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, stride, pad, act, residual, pool: one and several warps to a contraction, contractions shorter than a
    # warp's first loads and longer than several refills, ragged last pixel and filter tiles, windows that leave the image on
    # every side, pools over whole and partial tiles, a 3-channel layer, a contraction of 1134 pieces and one beyond the table of 1700
    (1, 3, 32, 32, 45, 3, 1, 1, "relu", False, None), (1, 8, 5, 5, 9, 1, 1, 0, "none", False, None), (1, 64, 1, 1, 300, 1, 1, 0, "relu6", True, None),
    (2, 207, 2, 2, 243, 3, 1, 1, "relu", False, "max2x2"), (1, 45, 30, 26, 58, 3, 1, 1, "relu6", False, "max2x2"), (3, 44, 17, 13, 64, 3, 1, 1, "relu", True, None),
    (1, 75, 15, 16, 130, 5, 2, 2, "relu", False, None), (2, 256, 14, 14, 358, 3, 2, 1, "relu", False, None), (1, 1000, 7, 7, 24, 3, 1, 1, "none", True, None),
    (1, 1536, 3, 3, 16, 3, 1, 1, "relu", False, None), (4, 432, 14, 14, 96, 1, 1, 0, "none", True, None), (1, 16, 9, 40, 20, 7, 1, 3, "relu", False, None)])
def test_few_pixel_tasks(cp, case):
    N, C, H, W, K, R, stride, pad, act, res, pool = case
    plan = check_task(cp, N, C, H, W, K, R, stride, pad, act=act, with_res=res, pool=pool)
    assert (plan.variant == 3) == (C < 1536) and (plan.variant != 3 or plan.workspace_bytes == 0)


@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, act, residual, pool, M tiles: whole images side by side (last tile ragged, images not square, filters of
    # one and two border pixels, two channel blocks, residual of two 64-filter groups, pooled), then tiles of image rows with
    # streamed filters, a filter row and a tap at a time, the last channel block of one MMA step
    (321, 24, 4, 4, 40, 3, "relu", False, None, 65), (129, 72, 7, 7, 72, 3, "none", True, None, 65), (193, 16, 7, 7, 24, 5, "relu6", False, None, 65),
    (331, 40, 3, 5, 16, 3, "relu", False, None, 67), (193, 20, 8, 8, 24, 3, "none", False, "max2x2", 65), (385, 136, 4, 4, 130, 3, "relu", True, None, 39),
    (10, 136, 28, 28, 120, 3, "relu", True, None, 70), (10, 40, 28, 28, 208, 5, "none", False, None, 70)])
def test_patch_tiles_of_whole_images_and_streamed_filter_rows(cp, case):
    N, C, H, W, K, R, act, res, pool, tiles = case
    plan = check_task(cp, N, C, H, W, K, R, 1, R // 2, act=act, with_res=res, pool=pool, kernel="tensor")
    assert plan.variant == 1 and plan.tiles_m == tiles


@pytest.mark.parametrize("case", [
    # N, C, H, K, act, residual, pool, filters of a tile (a multiple of 32 above the 16 that K needs: only pairs of thread blocks have those):
    # even and odd numbers of tiles (the second block of the last pair without one), one and several tiles per pair, a last residual
    # block of 32 filters, whole small images, the 2x2 pool, filters that stay and filters that are streamed
    (41, 72, 12, 203, "relu", True, None, 224), (41, 40, 16, 140, "none", False, None, 160), (75, 72, 16, 70, "relu6", True, None, 96),
    (150, 72, 7, 203, "none", True, None, 224), (41, 40, 16, 140, "relu", False, "max2x2", 160), (75, 200, 8, 140, "none", False, "max2x2", 160),
    (64, 131, 28, 203, "relu", False, None, 224)])
def test_patch_tiles_of_pairs_of_thread_blocks(cp, case):
    N, C, H, K, act, res, pool, tile_n = case
    plan = check_task(cp, N, C, H, H, K, 3, 1, 1, act=act, with_res=res, pool=pool)
    assert plan.variant == 1 and plan.tile_n == tile_n


def test_stems_on_the_patch_kernel(cp):
    # enough tiles for the patch kernel: the input is regrouped into 16-channel pixels (stride 1 and 2)
    plan = check_task(cp, 16, 3, 64, 64, 64, 7, 2, 3, kernel="tensor")
    assert plan.variant == 1 and plan.workspace_bytes > 0     # the workspace holds the regrouped input
    check_task(cp, 16, 3, 62, 60, 32, 3, 2, 1, act="relu6", kernel="tensor")
    check_task(cp, 24, 3, 32, 32, 45, 3, 1, 1, kernel="tensor")
    check_task(cp, 20, 4, 36, 28, 24, 5, 1, 2, act="none", kernel="tensor")


@pytest.mark.parametrize("case", [
    # N, H, W, K, R, stride, pad, act, pool: 1, 2 and 4 conv rows per step, images whose steps are dealt unevenly to the blocks
    # (with the pool: one conv row above recomputed), ragged last step, rows and columns outside the image on every side,
    # windows of 32, 64 and 128 bytes, filters that fill 32, 64 and 128 rows
    (9, 64, 64, 45, 3, 1, 1, "relu", None), (5, 224, 224, 32, 3, 2, 1, "relu6", None), (4, 64, 136, 64, 7, 2, 3, "relu", "max3x3s2"),
    (20, 32, 132, 48, 7, 2, 3, "relu6", "max3x3s2"), (9, 68, 76, 24, 5, 1, 2, "none", None), (17, 70, 132, 100, 5, 2, 2, "relu", None),
    (40, 63, 132, 8, 3, 2, 0, "none", None), (20, 36, 132, 40, 4, 2, 1, "none", "max3x3s2"), (9, 64, 68, 120, 3, 1, 1, "relu", None)])
def test_stems_straight_from_the_image(cp, case):
    N, H, W, K, R, stride, pad, act, pool = case
    x, w, b, _ = wl.conv_task_tensors(95, N, 3, H, W, K, R, R)
    plan = cp.cprune_task_plan(N, 3, H, W, K, R, R, stride, pad, 1, act, False, pool)
    packed, fc = cp.cprune_pack_weights(plan, _dev(w), _dev(b)), cp.cprune_fc_pack(torch.ones((8, K), device="cuda"))
    tasks = [cp.TaskDesc(op=cp.OP_CONV, in_=0, out=1, res=-1, plan=plan.handle, w=packed[0].data_ptr(), b=packed[1].data_ptr()),
             cp.TaskDesc(op=cp.OP_GAP, in_=1, out=2, res=-1),
             cp.TaskDesc(op=cp.OP_FC, in_=2, out=3, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=K, p1=8)]
    model = cp.cprune_model_create(N, H, W, 3, tasks, keep_alive=(plan, packed, fc))
    assert model.launches == 3
    cp.cprune_model_run(model, _dev(x))
    y = model.copy_tensor(1).float().cpu().numpy()
    cp.cprune_poll_device_status()
    ref, bound = _pooled(*oracle.conv2d(x, w, b, stride, pad, 1, act, None, with_bound=True), pool)
    rb = oracle.round_bf16
    ref_m, bound_m = _pooled(*oracle.conv2d(rb(x), rb(w), b, stride, pad, 1, act, None, with_bound=True), pool)
    assert y.shape[:3] == ref.shape[:3] and np.all(y[..., K:] == 0)
    check_values("stem %s" % (case,), y[..., :K], ref, bound, ref_m, bound_m)
    # an image that is not 16-byte aligned takes the bf16 copy; the same values up to the order of the sums
    odd = torch.empty(x.size + 1, device="cuda")[1:].view(x.shape)
    odd.copy_(_dev(x))
    cp.cprune_model_run(model, odd)
    y2 = model.copy_tensor(1).float().cpu().numpy()
    check_values("stem, unaligned image %s" % (case,), y2[..., :K], ref, bound, ref_m, bound_m)


def stem_model(cp, plan, w, b):
    """A model of one conv task that reads its float32 image, a pool and a small FC layer."""
    K = plan.K
    packed, fc = cp.cprune_pack_weights(plan, _dev(w), _dev(b)), cp.cprune_fc_pack(torch.ones((8, K), device="cuda"))
    tasks = [cp.TaskDesc(op=cp.OP_CONV, in_=0, out=1, res=-1, plan=plan.handle, w=packed[0].data_ptr(), b=packed[1].data_ptr()),
             cp.TaskDesc(op=cp.OP_GAP, in_=1, out=2, res=-1),
             cp.TaskDesc(op=cp.OP_FC, in_=2, out=3, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=K, p1=8)]
    model = cp.cprune_model_create(plan.N, plan.H, plan.W, 3, tasks, keep_alive=(plan, packed, fc))
    assert model.launches == 3          # the conv task reads the image itself
    return model


@pytest.mark.parametrize("case", [
    # N, H, W, K, R, stride, pad, act, pool: rows that leave room for one accumulator, windows read as pairs of floats (3, 5 and 7 wide)
    # and value by value (1, 6 and 8 wide; 18 and 24 values), one and two MMA steps a row, blocks of one to four steps;
    # pooled rows of 64 columns and of 8 filters
    (9, 40, 480, 32, 3, 2, 1, "relu6", None), (7, 41, 472, 24, 5, 2, 2, "none", None), (17, 70, 132, 100, 5, 2, 1, "relu", None),
    (9, 64, 68, 40, 6, 1, 2, "none", None), (9, 66, 140, 33, 8, 2, 3, "relu", None), (40, 64, 128, 16, 1, 2, 0, "none", None),
    (40, 32, 256, 64, 7, 2, 3, "relu", "max3x3s2"), (20, 32, 132, 8, 3, 2, 1, "none", "max3x3s2")])
def test_stems_with_every_kind_of_window(cp, case):
    N, H, W, K, R, stride, pad, act, pool = case
    x, w, b, _ = wl.conv_task_tensors(97, N, 3, H, W, K, R, R)
    plan = cp.cprune_task_plan(N, 3, H, W, K, R, R, stride, pad, 1, act, False, pool)
    model = stem_model(cp, plan, w, b)
    assert model.reads_image
    for _ in range(2):
        cp.cprune_model_run(model, _dev(x))
    y = model.copy_tensor(1).float().cpu().numpy()
    cp.cprune_poll_device_status()
    ref, bound = _pooled(*oracle.conv2d(x, w, b, stride, pad, 1, act, None, with_bound=True), pool)
    rb = oracle.round_bf16
    ref_m, bound_m = _pooled(*oracle.conv2d(rb(x), rb(w), b, stride, pad, 1, act, None, with_bound=True), pool)
    assert np.all(y[..., K:] == 0)
    check_values("stem %s" % (case,), y[..., :K], ref, bound, ref_m, bound_m)


@pytest.mark.parametrize("filters,bias", [(4, 0), (8, 0), (0, 1)])
def test_a_stem_from_the_image_refuses_misaligned_parameters(cp, filters, bias):
    # on the host, as the task by itself does: no kernel reads them
    plan = cp.cprune_task_plan(9, 3, 40, 480, 32, 3, 3, 2, 1)
    x, w, b, _ = wl.conv_task_tensors(98, 9, 3, 40, 480, 32, 3, 3)
    wp, bp = cp.cprune_pack_weights(plan, _dev(w), _dev(b))
    fc = cp.cprune_fc_pack(torch.ones((8, 32), device="cuda"))
    room = torch.zeros(wp.numel() * wp.element_size() + 16, dtype=torch.uint8, device="cuda")
    tasks = [cp.TaskDesc(op=cp.OP_CONV, in_=0, out=1, res=-1, plan=plan.handle, w=room.data_ptr() + filters if filters else wp.data_ptr(), b=bp.data_ptr() + bias),
             cp.TaskDesc(op=cp.OP_GAP, in_=1, out=2, res=-1),
             cp.TaskDesc(op=cp.OP_FC, in_=2, out=3, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=32, p1=8)]
    model = cp.cprune_model_create(9, 40, 480, 3, tasks, keep_alive=(plan, wp, bp, fc, room))
    assert model.reads_image
    with pytest.raises(cp.CpruneError) as e:
        cp.cprune_model_run(model, _dev(x))
    assert e.value.status == 1                        # CPRUNE_ERR_INVALID_ARG


@pytest.mark.parametrize("case", [
    # N, H, W, K, R, stride, pad, act: images too large for a step of 128 filter rows, so that a step has one or two conv rows of 32
    # or 64 filters and the other rows of the MMA go nowhere; two or three steps per block (both staging buffers), every step's bias
    # other than zero
    (4, 224, 224, 64, 7, 2, 3, "relu"), (3, 224, 224, 48, 7, 2, 3, "none"), (4, 160, 160, 24, 3, 1, 1, "relu6"),
    (2, 320, 320, 32, 3, 2, 1, "relu")])
def test_stems_of_large_images_with_fewer_conv_rows_per_step(cp, case):
    N, H, W, K, R, stride, pad, act = case
    x, w, b, _ = wl.conv_task_tensors(96, N, 3, H, W, K, R, R)
    plan = cp.cprune_task_plan(N, 3, H, W, K, R, R, stride, pad, 1, act)
    model = stem_model(cp, plan, w, b)
    for _ in range(2):
        cp.cprune_model_run(model, _dev(x))
    y = model.copy_tensor(1).float().cpu().numpy()
    cp.cprune_poll_device_status()
    ref, bound = oracle.conv2d(x, w, b, stride, pad, 1, act, None, with_bound=True)
    rb = oracle.round_bf16
    ref_m, bound_m = oracle.conv2d(rb(x), rb(w), b, stride, pad, 1, act, None, with_bound=True)
    assert np.all(y[..., K:] == 0)
    check_values("stem of a large image %s" % (case,), y[..., :K], ref, bound, ref_m, bound_m)


@pytest.mark.parametrize("case", [
    # N, H, W, K, R, stride, pad, act, pool: 1, 2 and 4 conv rows per step (two of them with rows of the MMA left over), windows of 32,
    # 64 and 128 bytes with one to thirteen pixels behind the filter's last
    (9, 64, 64, 45, 3, 1, 1, "none", None), (5, 224, 224, 32, 3, 2, 1, "none", None), (4, 160, 160, 24, 3, 1, 1, "relu6", None),
    (3, 224, 224, 48, 7, 2, 3, "none", None), (9, 68, 76, 24, 5, 1, 2, "relu", None), (9, 64, 68, 120, 3, 1, 1, "none", None),
    (20, 36, 132, 40, 4, 2, 1, "none", "max3x3s2"), (4, 64, 136, 64, 7, 2, 3, "relu", "max3x3s2")])
def test_a_pixel_that_is_no_number_reaches_only_the_conv_rows_whose_window_holds_it(cp, case):
    # conv rows of one step share their input rows and windows are stored wider than the filter: neither may be multiplied with zeros
    N, H, W, K, R, stride, pad, act, pool = case
    plan = cp.cprune_task_plan(N, 3, H, W, K, R, R, stride, pad, 1, act, False, pool)
    x, w, b, _ = wl.conv_task_tensors(99, N, 3, H, W, K, R, R)
    model = stem_model(cp, plan, w, b)
    bad, pixels = x.copy(), ((1, 21, 30, np.nan), (2, 38 % (H - 2), 61, np.inf))
    for n, h, v, value in pixels:
        bad[n, h, v, 1] = value
    out = []
    for t in (x, bad):
        cp.cprune_model_run(model, _dev(t))
        out.append(model.copy_tensor(1).float().cpu().numpy()[..., :K])
    cp.cprune_poll_device_status()
    touched = np.zeros((N, plan.P, plan.Q, 1))
    for n, h, v, _ in pixels:
        p, q = np.arange(plan.P) * stride - pad, np.arange(plan.Q) * stride - pad
        touched[n, ..., 0] = ((p <= h) & (h < p + R))[:, None] & ((q <= v) & (v < q + R))[None, :]
    if pool:
        touched = oracle.maxpool(touched, 3, 2, 1)
    touched = np.broadcast_to(touched > 0, out[0].shape)
    assert np.array_equal(out[0][~touched], out[1][~touched])
    if act != "none":
        assert np.all(np.isfinite(out[1][1])) and (pool or np.all(out[1][1][touched[1]] == 0))
    elif not pool:
        assert np.all(np.isnan(out[1][1][touched[1]])) and not np.any(np.isfinite(out[1][2][touched[2]]))


def test_the_task_times_of_a_model_are_those_of_the_kernels_it_launches(cp):
    # the entry of a first task that reads the image is timed on that kernel, with an image of zeros in the place of the unused bf16 copy
    N, H, K = 16, 128, 48
    plan = cp.cprune_task_plan(N, 3, H, H, K, 7, 7, 2, 3, 1)
    _, w, b, _ = wl.conv_task_tensors(102, 1, 3, 8, 8, K, 7, 7)
    model = stem_model(cp, plan, w, b)
    assert model.reads_image
    cp.cprune_model_run(model, torch.zeros((N, H, H, 3), device="cuda"))
    a = model.copy_tensor(1)
    mark = _dev(np.full((N, H, H, 3), 7.0, dtype=np.float32))
    ptr, _ = model.tensor(0)
    assert cp.lib().cprune_cast_input(mark.data_ptr(), N * H * H, 3, ptr, torch.cuda.current_stream().cuda_stream) == 0
    (ms,) = model.time_tasks(2)
    cp.cprune_poll_device_status()
    assert torch.equal(model.copy_tensor(1), a) and 0 < ms < 5


def test_passes_with_new_images_and_newly_packed_filters_follow_each_other_unwaited(cp):
    # a chain of three short kernels: a pass must see the parameters that the kernel just before it packed, and nothing of the
    # images of the passes before it
    N, H, K = 9, 64, 45
    plan = cp.cprune_task_plan(N, 3, H, H, K, 3, 3, 1, 1, 1)
    xs = [_dev(wl.conv_task_tensors(104 + j, N, 3, H, H, K, 3, 3)[0]) for j in range(3)]
    ws = [[_dev(t) for t in wl.conv_task_tensors(107 + j, N, 3, 8, 8, K, 3, 3)[1:3]] for j in range(2)]
    fc = cp.cprune_fc_pack(_dev(wl.normal_f32(109, 0, (8, K))))
    packed = cp.cprune_pack_weights(plan, *ws[0])
    tasks = [cp.TaskDesc(op=cp.OP_CONV, in_=0, out=1, res=-1, plan=plan.handle, w=packed[0].data_ptr(), b=packed[1].data_ptr()),
             cp.TaskDesc(op=cp.OP_GAP, in_=1, out=2, res=-1),
             cp.TaskDesc(op=cp.OP_FC, in_=2, out=3, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=K, p1=8)]
    model = cp.cprune_model_create(N, H, H, 3, tasks, keep_alive=(plan, packed, fc))
    assert model.reads_image
    st = torch.cuda.current_stream().cuda_stream

    def passes(wait):
        out = []
        for i in range(24):
            if i % 4 == 0:
                w, b = ws[i // 4 % 2]
                assert cp.lib().cprune_pack_weights(plan.handle, w.data_ptr(), b.data_ptr(), packed[0].data_ptr(), packed[1].data_ptr(), st) == 0
            if wait:
                torch.cuda.synchronize()
            out.append(cp.cprune_model_run(model, xs[i % 3]))
        torch.cuda.synchronize()
        return out

    want = passes(True)
    assert not torch.equal(want[0], want[1]) and not torch.equal(want[0], want[12])
    for _ in range(20):
        for a, b in zip(passes(False), want):
            assert torch.equal(a, b)
    cp.cprune_poll_device_status()


def test_a_first_task_that_adds_the_image_to_its_result(cp):
    # the residual is the bf16 copy of the image: it has to be made even where the convolution itself runs on a regrouped input
    N, H = 64, 128
    plan = cp.cprune_task_plan(N, 3, H, H, 3, 3, 3, 1, 1, 1, "none", True)
    x, w, b, _ = wl.conv_task_tensors(103, N, 3, H, H, 3, 3, 3)
    packed, fc = cp.cprune_pack_weights(plan, _dev(w), _dev(b)), cp.cprune_fc_pack(torch.ones((8, 3), device="cuda"))
    tasks = [cp.TaskDesc(op=cp.OP_CONV, in_=0, out=1, res=0, plan=plan.handle, w=packed[0].data_ptr(), b=packed[1].data_ptr()),
             cp.TaskDesc(op=cp.OP_GAP, in_=1, out=2, res=-1),
             cp.TaskDesc(op=cp.OP_FC, in_=2, out=3, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=3, p1=8)]
    model = cp.cprune_model_create(N, H, H, 3, tasks, keep_alive=(plan, packed, fc))
    cp.cprune_model_run(model, _dev(x))
    xb = cp.cprune_cast_input(_dev(x))
    assert plan.variant == 1 and torch.equal(model.copy_tensor(1), cp.cprune_task_run(plan, xb, *packed, xb))


def test_an_image_off_a_16_byte_boundary_is_cast_and_regrouped_in_one_pass(cp):
    N, H, K = 16, 128, 64
    plan = cp.cprune_task_plan(N, 3, H, H, K, 7, 7, 2, 3, 1)
    assert plan.variant == 1 and plan.workspace_bytes > 0           # by itself the task runs on a regrouped input
    x, w, b, _ = wl.conv_task_tensors(101, N, 3, H, H, K, 7, 7)
    model = stem_model(cp, plan, w, b)
    mark = _dev(np.full((N, H, H, 3), 7.0, dtype=np.float32))
    ptr, _ = model.tensor(0)                                        # the bf16 copy of the image, which nobody needs
    assert cp.lib().cprune_cast_input(mark.data_ptr(), N * H * H, 3, ptr, torch.cuda.current_stream().cuda_stream) == 0
    odd = torch.empty(x.size + 1, device="cuda")[1:].view(x.shape)
    odd.copy_(_dev(x))
    cp.cprune_model_run(model, odd)
    a = model.copy_tensor(1)
    assert torch.all(model.copy_tensor(0)[..., :3] == 7.0)
    y = cp.cprune_task_run(plan, cp.cprune_cast_input(_dev(x)), *cp.cprune_pack_weights(plan, _dev(w), _dev(b)))
    cp.cprune_poll_device_status()
    assert torch.equal(a, y)                                        # the task's own kernel on the same values


@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, stride, pad: fused in the patch kernel (tiles around whole 3x3 windows, even and odd extents),
    # and as a separate pass (few tiles; a task with wrap-around slots)
    (16, 3, 64, 64, 64, 7, 2, 3), (12, 3, 60, 52, 40, 7, 2, 3), (40, 3, 30, 30, 24, 3, 1, 1),
    (2, 3, 64, 64, 64, 7, 2, 3), (2, 16, 30, 30, 24, 3, 1, 1)])
def test_maxpool_3x3_stride_2(cp, case):
    N, C, H, W, K, R, stride, pad = case
    plan = check_task(cp, N, C, H, W, K, R, stride, pad, act="relu", pool="max3x3s2", kernel="tensor")
    P = oracle.out_size(H, R, stride, pad)
    assert plan.out_h == (P - 1) // 2 + 1


def test_maxpool_3x3_stride_2_pooled_by_the_epilogue_warps(cp):
    # the fused pool normally runs on separate pooling warps; a plan flag selects the instantiation in which the epilogue
    # warps pool the tile themselves, which plans with one staging buffer use
    check_task(cp, 16, 3, 64, 64, 64, 7, 2, 3, act="relu", pool="max3x3s2", kernel="tensor", flags=("pool_on_epilogue_warps",))
    check_task(cp, 40, 3, 30, 30, 24, 3, 1, 1, act="none", pool="max3x3s2", kernel="tensor", flags=("pool_on_epilogue_warps",))
    check_task(cp, 40, 3, 30, 30, 24, 3, 1, 1, act="none", pool="max3x3s2", kernel="tensor")


def test_stride_1_tasks_on_the_im2col_kernel(cp):
    # the im2col kernel serves stride-1 tasks too when a plan asks for it (and whenever the patch kernel declines)
    for case in ((16, 64, 32, 32, 48, 3, 1, 1), (8, 130, 14, 14, 260, 3, 1, 1), (8, 24, 56, 56, 108, 1, 1, 0)):
        plan = check_task(cp, *case, kernel="tensor", flags=("im2col_only",))
        assert plan.variant == 0


def big_task_tensors(seed, N, C, H, W, K, R, groups, with_res, P, Q, base=4):
    """Tensors of a full-size task (drawing every image from the generator would take minutes over a whole model)."""
    return wl.conv_task_tensors_tiled(seed, N, C, H, W, K, R, R, groups, with_res, P, Q, base)


def sample_points(rng, N, oh, ow, K, n_pts):
    pts = np.stack([rng.integers(0, N, n_pts), rng.integers(0, oh, n_pts), rng.integers(0, ow, n_pts),
                    rng.integers(0, K, n_pts)], axis=1)
    # corners and edges are where padding, ragged tiles and pooling windows go wrong
    pts[:8, 1:3] = [[0, 0], [0, ow - 1], [oh - 1, 0], [oh - 1, ow - 1], [0, ow // 2], [oh // 2, 0], [oh - 1, ow // 2], [oh // 2, ow - 1]]
    pts[:4, 0] = [0, N - 1, 0, N - 1]
    pts[8:12, 3] = [0, K - 1, K // 2, max(K - 2, 0)]
    return pts


def points_reference(x, w, b, stride, pad, groups, act, res, pool, pts, P, Q):
    """Oracle values and error scales at sampled OUTPUT coordinates (after the optional pool)."""
    if pool is None:
        return oracle.conv2d_points(x, w, b, stride, pad, groups, act, res, pts)
    win, st, off = (3, 2, 1) if pool == "max3x3s2" else (2, 2, 0)
    ref = np.full(len(pts), -np.inf)
    bound = np.zeros(len(pts))
    for di in range(win):
        for dj in range(win):
            q = pts.copy()
            q[:, 1] = st * pts[:, 1] - off + di
            q[:, 2] = st * pts[:, 2] - off + dj
            inside = (q[:, 1] >= 0) & (q[:, 1] < P) & (q[:, 2] >= 0) & (q[:, 2] < Q)
            v, bd = oracle.conv2d_points(x, w, b, stride, pad, groups, act, res, q[inside])
            ref[inside] = np.maximum(ref[inside], v)
            bound[inside] = np.maximum(bound[inside], bd)
    return ref, bound


def check_task_sampled(cp, label, N, C, H, W, K, R, stride, pad, groups, act, with_res, pool, seed, n_pts=160, tensors=None):
    P, Q = oracle.out_size(H, R, stride, pad), oracle.out_size(W, R, stride, pad)
    x, w, b, res = tensors if tensors is not None else big_task_tensors(seed, N, C, H, W, K, R, groups, with_res, P, Q)
    y, plan = run_task(cp, x, w, b, stride, pad, groups, act, res, pool)
    pts = sample_points(np.random.default_rng(seed), N, plan.out_h, plan.out_w, K, n_pts)
    ref, bound = points_reference(x, w, b, stride, pad, groups, act, res, pool, pts, P, Q)
    rb = oracle.round_bf16
    ref_m, bound_m = points_reference(rb(x), rb(w), b, stride, pad, groups, act, None if res is None else rb(res), pool, pts, P, Q)
    got = y[pts[:, 0], pts[:, 1], pts[:, 2], pts[:, 3]]
    check_values(label, got, ref, bound, ref_m, bound_m)
    assert np.all(y[..., K:] == 0)
    return plan


def model_tasks(name, batch):
    """The distinct conv tasks of a pruned model as the pipeline plans them: (key, layer names)."""
    table = wl.MODELS[name]()
    m = wl.pruned_shapes(table)
    sz = wl.spatial_sizes(m)
    layers = m["layers"]
    readers = {}
    for l in layers:
        for key in ("in", "res"):
            if l.get(key) is not None:
                readers.setdefault(l[key], []).append(l["name"])
    out = {}
    for a, nxt in zip(layers, layers[1:] + [None]):
        if a["kind"] != "conv":
            continue
        pool = a.get("pool")
        if (nxt is not None and nxt["kind"] == "maxpool" and nxt["in"] == a["out"] and pool is None and a.get("res") is None
                and (nxt["k"], nxt["stride"], nxt["pad"]) == (3, 2, 1) and readers.get(a["out"]) == [nxt["name"]]):
            pool = "max3x3s2"           # the pipeline folds such a pool into the task
        h, w = sz[a["in"]]
        key = (batch, a["C"], h, w, a["K"], a["R"], a["stride"], a["pad"], a["groups"] if a["groups"] > 1 else 1, a["act"],
               a.get("res") is not None, pool)
        out.setdefault(key, []).append(a["name"])
    return out


BENCH_MODELS = [("resnet18", 64), ("mobilenet_v2", 64), ("vgg16_cifar", 128), ("resnet18", 1), ("mobilenet_v2", 1), ("vgg16_cifar", 1)]


@pytest.mark.parametrize("name,batch", BENCH_MODELS)
def test_every_plan_of_the_benchmarked_models_on_sampled_outputs(cp, name, batch):
    # every distinct task of the pruned model at the batch bench.py times it with, i.e. the very plans (tiles, split
    # reductions, kernel variants) of the benchmark, each checked on sampled outputs
    tasks = model_tasks(name, batch)
    families = {}
    for n_task, (key, names) in enumerate(tasks.items()):
        N, C, H, W, K, R, stride, pad, groups, act, with_res, pool = key
        plan = check_task_sampled(cp, "%s b%d %s" % (name, batch, names[0]), N, C, H, W, K, R, stride, pad, groups, act, with_res,
                                  pool, seed=100 + n_task)
        fam = cp.KERNEL_NAMES[plan.kernel]
        assert fam == ("depthwise" if groups > 1 else "tensor"), (names, fam)      # no dense task falls off the tensor cores
        families[names[0]] = (fam, plan.variant, plan.splits, plan.tile_m, plan.tile_n)
    print("\n%s batch %d: %d distinct tasks" % (name, batch, len(tasks)))
    for k, v in families.items():
        print("  %-14s %s variant %d splits %d tile %dx%d" % ((k,) + v))
    if (name, batch) == ("resnet18", 64):
        assert len(tasks) == 15
        assert families["stem"][1] == 1 and families["l1b1_conv1"][1] == 1 and families["l3b1_conv2"][1] == 1
    if (name, batch) == ("mobilenet_v2", 64):
        assert len(tasks) == 30
        assert families["b2_exp"][1] in (1, 2) and families["b3_proj"][1] in (1, 2)


def sweep_keep_counts(k_full):
    """Kept filter counts checked per swept shape: full width, one less, and every 16 n +- 1 down to a quarter."""
    lo = (k_full + 3) // 4
    ks = {k_full, k_full - 1, lo}
    for n in range(k_full // 16 + 1):
        for k in (16 * n - 1, 16 * n + 1):
            if lo <= k <= k_full:
                ks.add(k)
    return sorted(k for k in ks if k >= 1)


def test_sweep_parity_over_the_kept_filter_count(cp):
    # every distinct conv shape of the models, with the filters that L1 selection keeps at each checked count (for
    # depthwise shapes the input channels go with the filters), at batch 2 on sampled outputs
    n_points = 0
    for si, shp in enumerate(wl.sweep_shapes()):
        dw = shp["groups"] > 1
        R, stride, pad, act = shp["R"], shp["stride"], shp["pad"], shp["act"]
        P, Q = oracle.out_size(shp["H"], R, stride, pad), oracle.out_size(shp["W"], R, stride, pad)
        x, w, b, _ = wl.conv_task_tensors(500 + si, 2, shp["C"], shp["H"], shp["W"], shp["K"], R, R, shp["groups"])
        for K in sweep_keep_counts(shp["K"]):
            kept = oracle.select_indices(w, K)
            xs = np.ascontiguousarray(x[..., kept]) if dw else x
            label = "sweep %s/%s" % (shp["model"], shp["layer"])
            plan = check_task_sampled(cp, label, 2, K if dw else shp["C"], shp["H"], shp["W"], K, R, stride, pad, K if dw else 1, act,
                                      False, None, seed=si * 1000 + K, n_pts=64, tensors=(xs, w[kept], b[kept], None))
            assert cp.KERNEL_NAMES[plan.kernel] == ("depthwise" if dw else "tensor")
            n_points += 1
    assert n_points > 800


@pytest.mark.parametrize("batch", [64, 1])
def test_sweep_parity_at_the_benchmarked_batches(cp, batch):
    # the sweep's own launch configurations: every shape at three kept counts (full, about 60 %, a quarter)
    for si, shp in enumerate(wl.sweep_shapes()):
        dw = shp["groups"] > 1
        R, stride, pad, act = shp["R"], shp["stride"], shp["pad"], shp["act"]
        P, Q = oracle.out_size(shp["H"], R, stride, pad), oracle.out_size(shp["W"], R, stride, pad)
        x, w, b, _ = big_task_tensors(700 + si, batch, shp["C"], shp["H"], shp["W"], shp["K"], R, shp["groups"], False, P, Q, base=2)
        for K in sorted({shp["K"], (3 * shp["K"]) // 5 + 1, (shp["K"] + 3) // 4}):
            kept = oracle.select_indices(w, K)
            xs = np.ascontiguousarray(x[..., kept]) if dw else x
            check_task_sampled(cp, "sweep b%d %s/%s" % (batch, shp["model"], shp["layer"]), batch, K if dw else shp["C"], shp["H"],
                               shp["W"], K, R, stride, pad, K if dw else 1, act, False, None, seed=si * 1000 + K, n_pts=64,
                               tensors=(xs, w[kept], b[kept], None))


@pytest.mark.parametrize("C", [64, 65, 66, 67, 68, 69, 70, 71, 72, 73, 79, 80, 81])
def test_every_channel_residue(cp, C):
    # C and K sweep the residues modulo 8 and 16 around a 64-channel block boundary
    check_task(cp, 1, C, 10, 10, C + 3, 3, 1, 1, kernel="tensor")


@pytest.mark.parametrize("kernel", ["tensor", "direct"])
def test_three_channel_stems(cp, kernel):
    # 3 input channels: the tensor-core kernel packs 8 taps x 8 padded channels into one K block
    plan = check_task(cp, 1, 3, 32, 32, 45, 3, 1, 1, kernel=kernel)
    assert cp.KERNEL_NAMES[plan.kernel] == kernel
    check_task(cp, 1, 3, 37, 37, 64, 7, 2, 3, kernel=kernel)
    check_task(cp, 2, 3, 30, 30, 32, 3, 2, 1, act="relu6", kernel=kernel)
    check_task(cp, 3, 3, 64, 64, 64, 7, 2, 3, kernel=kernel)
    check_task(cp, 2, 5, 21, 19, 24, 5, 1, 2, kernel=kernel)
    assert cp.KERNEL_NAMES[cp.cprune_task_plan(1, 3, 224, 224, 64, 7, 7, 2, 3).kernel] == "tensor"


@pytest.mark.parametrize("C,H,W,stride", [(32, 16, 16, 1), (72, 15, 17, 2), (108, 14, 14, 1), (144, 7, 9, 2),
                                          (8, 5, 5, 1), (432, 14, 14, 2), (720, 7, 7, 1), (20, 3, 2, 1)])
def test_depthwise_task_parity(cp, C, H, W, stride):
    plan = check_task(cp, 2, C, H, W, C, 3, stride, 1, groups=C, act="relu6")
    assert cp.KERNEL_NAMES[plan.kernel] == "depthwise"


@pytest.mark.parametrize("C,H,W,stride", [(72, 56, 56, 2), (120, 28, 28, 1), (90, 17, 15, 2), (576, 14, 14, 2), (1152, 7, 7, 1),
                                          (8, 6, 5, 1), (20, 3, 2, 1)])
def test_depthwise_5x5_task_parity(cp, C, H, W, stride):
    # MnasNet's 5x5 depthwise layers (pad 2): ragged tiles, channel counts off the 8 / 64 grid, images smaller than the filter
    plan = check_task(cp, 2, C, H, W, C, 5, stride, 2, groups=C, act="relu")
    assert cp.KERNEL_NAMES[plan.kernel] == "depthwise"
    check_task(cp, 1, C, H, W, C, 5, stride, 2, groups=C, act="none", with_res=(stride == 1))


@pytest.mark.parametrize("N,C,H,W,R,stride,res", [(40, 20, 57, 55, 3, 1, False), (40, 200, 29, 31, 3, 2, False), (26, 72, 33, 61, 5, 1, True),
                                                  (30, 136, 23, 40, 5, 2, False), (1, 8, 1, 1, 3, 1, False), (1, 72, 40, 2, 5, 1, False)])
def test_depthwise_tiles_of_a_persistent_block(cp, N, C, H, W, R, stride, res):
    # several tiles per thread block (both patch buffers refilled), odd extents against the two-column strips and the row
    # segments, a last channel block that is not full, and images smaller than a strip or a segment
    check_task(cp, N, C, H, W, C, R, stride, R // 2, groups=C, act="relu6", with_res=res)


def test_task_runs_are_deterministic(cp):
    x, w, b, _ = wl.conv_task_tensors(5, 2, 89, 14, 14, 128, 3, 3)
    plan = cp.cprune_task_plan(2, 89, 14, 14, 128, 3, 3, 1, 1)
    xb = cp.cprune_cast_input(_dev(x))
    wp, bp = cp.cprune_pack_weights(plan, _dev(w), _dev(b))
    a = cp.cprune_task_run(plan, xb, wp, bp).clone()
    c = cp.cprune_task_run(plan, xb, wp, bp)
    cp.cprune_poll_device_status()
    assert torch.equal(a, c)


@pytest.mark.parametrize("case", [(1, 64, 14, 14, 96, 3, 1, 1), (4, 96, 14, 14, 576, 1, 1, 0), (2, 128, 28, 28, 256, 3, 2, 1)])
def test_channel_subset_property_on_the_gpu(cp, case):
    # pruning to any K gives the same values as the matching channels of the full-width task: one full-width check
    # therefore vouches for every K of a sweep whose plans accumulate in the same order
    N, C, H, W, K, R, stride, pad = case
    x, w, b, _ = wl.conv_task_tensors(6, N, C, H, W, K, R, R)
    full, _ = run_task(cp, x, w, b, stride, pad)
    for keep in (K // 4, K // 3 + 5, (3 * K) // 4, K - 1):
        kept = oracle.select_indices(w, keep)
        y, _ = run_task(cp, x, w[kept], b[kept], stride, pad)
        assert np.array_equal(y[..., :keep], full[..., kept]), keep


def test_task_argument_errors(cp):
    bad = [dict(N=0), dict(C=-1), dict(stride=0), dict(pad=-1), dict(R=40, S=40)]
    base = dict(N=1, C=8, H=8, W=8, K=8, R=3, S=3, stride=1, pad=1)
    for chg in bad:
        a = dict(base, **chg)
        with pytest.raises(cp.CpruneError) as e:
            cp.cprune_task_plan(a["N"], a["C"], a["H"], a["W"], a["K"], a["R"], a["S"], a["stride"], a["pad"])
        assert e.value.status == 1
    with pytest.raises(cp.CpruneError) as e:
        cp.cprune_task_plan(1, 8, 8, 8, 16, 3, 3, 1, 1, groups=2)
    assert e.value.status == 2
    plan = cp.cprune_task_plan(1, 8, 8, 8, 8, 3, 3, 1, 1, residual=True)
    xb = torch.zeros((1, 8, 8, 8), dtype=torch.bfloat16, device="cuda")
    wp, bp = cp.cprune_pack_weights(plan, torch.zeros((8, 8, 3, 3), device="cuda"), torch.zeros(8, device="cuda"))
    with pytest.raises(cp.CpruneError) as e:
        cp.cprune_task_run(plan, xb, wp, bp, None)          # the plan wants a residual
    assert e.value.status == 1


# ------------------------------------------------------------------ tail operators

def test_cast_pool_gap_fc(cp):
    x = wl.normal_f32(31, 0, (2, 9, 11, 13))
    xb = cp.cprune_cast_input(_dev(x))
    got = xb.float().cpu().numpy()
    assert np.array_equal(got[..., :13], oracle.round_bf16(x)) and np.all(got[..., 13:] == 0)
    xr = oracle.round_bf16(x)
    for k, s, p in ((3, 2, 1), (2, 2, 0)):
        y = cp.cprune_maxpool(xb, 13, k, s, p).float().cpu().numpy()
        assert np.array_equal(y[..., :13], oracle.maxpool(xr, k, s, p))
    g = cp.cprune_global_avgpool(xb, 13).float().cpu().numpy()
    ref = oracle.gap(xr)
    assert np.max(np.abs(g[:, :13] - ref)) <= 2.0 ** -8 * np.max(np.abs(ref)) + 1e-6
    a = wl.normal_f32(31, 1, (5, 243))
    w = wl.normal_f32(31, 2, (37, 243), 0.1)
    b = wl.normal_f32(31, 3, (37,), 0.1)
    ab = cp.cprune_cast_input(_dev(a))
    wp, bp = cp.cprune_fc_pack(_dev(w), _dev(b))
    ref, bound = oracle.fc(a, w, b, "relu", with_bound=True)
    y32 = cp.cprune_fc(ab, 243, wp, bp, 37, "relu", out_f32=True).cpu().numpy()
    assert np.max(np.abs(y32 - ref) / bound) <= TOL
    y16 = cp.cprune_fc(ab, 243, wp, bp, 37, "relu").float().cpu().numpy()
    assert np.max(np.abs(y16[:, :37] - ref) / bound) <= TOL and np.all(y16[:, 37:] == 0)
    assert np.array_equal(cp.cprune_widen_output(ab).cpu().numpy(), ab.float().cpu().numpy())


# ------------------------------------------------------------------ whole models

def model_parity(cp, name, batch, hw=None, kernel="auto", oracle_images=None):
    """The whole pruned network on `batch` images against the oracle on the first `oracle_images` of them (images are
    independent; the plans are those of the full batch)."""
    from paper_2207_01260_b200.pipeline import PrunedNetwork
    table = wl.MODELS[name]()
    if hw:
        table["input"] = (hw, hw, table["input"][2])
    weights = wl.model_weights(table)
    x = wl.model_input(table, batch)
    net = PrunedNetwork(table, weights, batch, kernel=kernel)
    cp.cprune_poll_device_status()
    pw, kept = oracle.prune_model(table, weights)
    for lname, idx in kept.items():                     # selection is bit-exact, layer by layer
        assert np.array_equal(net.kept[lname].cpu().numpy(), idx), lname
    for lname, (w, b) in pw.items():
        gw, gb = net.params[lname]
        assert gw.cpu().numpy().tobytes() == w.tobytes() and gb.cpu().numpy().tobytes() == b.tobytes(), lname
    logits = net.run(_dev(x))
    cp.cprune_poll_device_status()
    logits2 = net.run(_dev(x), use_graph=True)
    logits3 = net.run(_dev(x), use_graph=True).clone()
    cp.cprune_poll_device_status()
    got = logits.cpu().numpy()
    assert np.array_equal(got, logits2.cpu().numpy()) and np.array_equal(got, logits3.cpu().numpy())
    # the host-buffer entry point (copies inside the call, two alternating device buffers)
    xh = torch.from_numpy(np.ascontiguousarray(x)).pin_memory()
    lh = torch.empty(got.shape, dtype=torch.float32).pin_memory()
    for _ in range(3):
        net.run_host(xh, lh)
    torch.cuda.synchronize()
    cp.cprune_poll_device_status()
    assert np.array_equal(lh.numpy(), got)
    n_ref = batch if oracle_images is None else min(batch, oracle_images)
    got = got[:n_ref]
    matched = oracle.model_ref(table, pw, x[:n_ref], matched=True)
    exact = oracle.model_ref(table, pw, x[:n_ref], matched=False)
    rel = np.linalg.norm(got - matched) / np.linalg.norm(matched)
    rel_exact = np.linalg.norm(got - exact) / np.linalg.norm(exact)
    assert rel <= 1e-2, (name, rel, rel_exact)
    # Top-1 must agree on every image whose answer is decided a priori: the oracle's top-2 gap exceeds twice the error
    # the tolerance allows a logit (1e-2 of the image's largest logit).  Images inside that margin have several correct
    # answers (random-weight networks have near-tied logits); they are counted, not judged.
    srt = np.sort(matched, axis=1)
    gap = srt[:, -1] - srt[:, -2]
    margin = 2.0 * 1e-2 * np.max(np.abs(matched), axis=1)
    decided = gap > margin
    agree = np.argmax(got, 1) == np.argmax(matched, 1)
    print("\n%s batch %d (%d images checked): rel-L2 %.2e matched / %.2e exact; top-1 agreement %d/%d raw, %d/%d decided a priori"
          % (name, batch, n_ref, rel, rel_exact, agree.sum(), n_ref, (agree & decided).sum(), decided.sum()))
    assert np.all(agree[decided]), np.nonzero(decided & ~agree)
    assert decided.mean() >= 0.25 or n_ref < 4, "too many near-ties to say anything"
    return net, rel, rel_exact


def test_vgg16_cifar_parity(cp):
    model_parity(cp, "vgg16_cifar", 4)
    model_parity(cp, "vgg16_cifar", 1, kernel="direct")


def test_resnet18_parity(cp):
    net, _, _ = model_parity(cp, "resnet18", 2)
    kinds = {cp.KERNEL_NAMES[i["kernel"]] for i in net.conv_launch_info().values()}
    assert kinds == {"tensor"}


def test_mobilenet_v2_parity(cp):
    net, _, _ = model_parity(cp, "mobilenet_v2", 2)
    kinds = {cp.KERNEL_NAMES[i["kernel"]] for i in net.conv_launch_info().values()}
    assert kinds == {"tensor", "depthwise"}


@pytest.mark.parametrize("name,batch,oracle_images", [("resnet18", 64, 12), ("mobilenet_v2", 64, 12), ("vgg16_cifar", 128, 32),
                                                      ("vgg16_cifar", 1, 1), ("resnet18", 1, 1), ("mobilenet_v2", 1, 1)])
def test_model_parity_at_the_benchmarked_batch(cp, name, batch, oracle_images):
    net, _, _ = model_parity(cp, name, batch, oracle_images=oracle_images)
    kinds = {cp.KERNEL_NAMES[i["kernel"]] for i in net.conv_launch_info().values()}
    assert "direct" not in kinds


def test_mnasnet_parity(cp):
    net, _, _ = model_parity(cp, "mnasnet1_0", 2)
    kinds = {cp.KERNEL_NAMES[i["kernel"]] for i in net.conv_launch_info().values()}
    assert kinds == {"tensor", "depthwise"}
    assert {net.plans[n].R for n in net.plans if n.endswith("_dw")} == {3, 5}
    model_parity(cp, "mnasnet1_0", 16, hw=96, oracle_images=4)


@pytest.mark.parametrize("N,inn,out,act", [(1, 3, 1, "none"), (16, 40, 10, "relu"), (17, 243, 130, "none"), (33, 1300, 24, "relu6"), (70, 2600, 9, "none")])
def test_fully_connected_tiles(cp, N, inn, out, act):
    # edges of the 16- and 32-image tiles, of the eight-feature blocks and of the input pieces dealt to eight warps (fewer than
    # one piece each, several rounds); float32 sums of exact bf16 products against float64: error far below 1e-5 of the scale
    x, w, b = wl.normal_f32(91, 0, (N, inn)), wl.normal_f32(91, 1, (out, inn), 0.1), wl.normal_f32(91, 2, (out,), 0.05)
    xb = cp.cprune_cast_input(_dev(x.reshape(N, 1, 1, inn))).reshape(N, -1)
    y = cp.cprune_fc(xb, inn, *cp.cprune_fc_pack(_dev(w), _dev(b)), out, act, out_f32=True).cpu().numpy()
    xr, wr = oracle.round_bf16(x).astype(np.float64), oracle.round_bf16(w).astype(np.float64)
    ref, scale = xr @ wr.T + b, np.abs(xr) @ np.abs(wr).T + np.abs(b)
    if act != "none":
        ref = np.clip(ref, 0, 6 if act == "relu6" else None)
    assert np.max(np.abs(y - ref) / scale) <= 1e-5


@pytest.mark.parametrize("N,inn,out", [(1, 512, 1000), (64, 358, 1000), (64, 512, 1000), (16, 1280, 1000), (64, 4096, 200), (8, 25088, 200)])
def test_fully_connected_sums_are_as_exact_as_float32_additions(cp, N, inn, out):
    # Relative error of the float32 results, 2-norm: the last rounding (at most 2^-24 of each value) and the running sums of a
    # warp, n = inn / 256 rounded additions.  Addition k of n rounds a partial sum of sqrt(k / n) of an eighth of the variance
    # by 0.43 * 2^-24 (rms), which makes (0.43 * 2^-24)^2 * n / 2 for the eight warps together: below (2^-24)^2 * n / 8.
    bound = 2.0 ** -24 * np.sqrt(1 + inn / 256 / 8)
    for positive in (True, False):
        x, w, b = wl.normal_f32(94, 0, (N, inn)), wl.normal_f32(94, 1, (out, inn), 1 / np.sqrt(inn)), wl.normal_f32(94, 2, (out,), 0.01)
        x = np.abs(x) if positive else x
        xb = cp.cprune_cast_input(_dev(x.reshape(N, 1, 1, inn))).reshape(N, -1)
        y = cp.cprune_fc(xb, inn, *cp.cprune_fc_pack(_dev(w), _dev(b)), out, "none", out_f32=True).cpu().numpy().astype(np.float64)
        ref = oracle.round_bf16(x).astype(np.float64) @ oracle.round_bf16(w).astype(np.float64).T + b
        rel = np.linalg.norm(y - ref) / np.linalg.norm(ref)
        assert rel <= bound, (rel, bound)


@pytest.mark.parametrize("N,inn,out,act", [(2369, 24, 8, "none"), (161, 72, 120, "relu"), (300, 1290, 130, "none")])
def test_fully_connected_tiles_of_sixteen_features(cp, N, inn, out, act):
    # more tiles of eight features than the GPU has SMs: the second eight beyond the padded output, half of the last tile, several
    # rounds of input pieces; the values are those of a small call, whose tiles have eight features, bit by bit
    x, w, b = wl.normal_f32(92, 0, (N, inn)), wl.normal_f32(92, 1, (out, inn), 0.1), wl.normal_f32(92, 2, (out,), 0.05)
    xb = cp.cprune_cast_input(_dev(x.reshape(N, 1, 1, inn))).reshape(N, -1)
    packed = cp.cprune_fc_pack(_dev(w), _dev(b))
    for f32 in (True, False):
        y = cp.cprune_fc(xb, inn, *packed, out, act, out_f32=f32)
        for n0 in (0, N // 16 * 16, 16):
            n1 = min(N, n0 + 16)
            assert torch.equal(y[n0:n1], cp.cprune_fc(xb[n0:n1].contiguous(), inn, *packed, out, act, out_f32=f32))


@pytest.mark.parametrize("N,inn,out,act", [(2353, 72, 24, "none"), (2369, 40, 40, "relu"), (700, 768, 130, "none"), (700, 1290, 136, "none"), (1100, 1290, 136, "none"),
                                           (1100, 4090, 120, "none"), (1100, 4100, 130, "relu")])
def test_fully_connected_grids_of_many_blocks(cp, N, inn, out, act):
    # more than 296 blocks of 16 features by 16 images, up to 768 and 4096 input features and beyond, two and three rounds of blocks: the values are those of a small call, bit by bit
    x, w, b = wl.normal_f32(94, 0, (N, inn)), wl.normal_f32(94, 1, (out, inn), 0.1), wl.normal_f32(94, 2, (out,), 0.05)
    xb = cp.cprune_cast_input(_dev(x.reshape(N, 1, 1, inn))).reshape(N, -1)
    packed = cp.cprune_fc_pack(_dev(w), _dev(b))
    for f32 in (True, False):
        y = cp.cprune_fc(xb, inn, *packed, out, act, out_f32=f32)
        for n0 in (0, 16, N // 32 * 16, N // 16 * 16 if N % 16 else N - 16):
            n1 = min(N, n0 + 16)
            assert torch.equal(y[n0:n1], cp.cprune_fc(xb[n0:n1].contiguous(), inn, *packed, out, act, out_f32=f32))


@pytest.mark.parametrize("hw", [(1, 1), (1, 7), (8, 8), (5, 13), (9, 14), (16, 17)])
def test_global_average_over_one_and_several_rounds_of_loads(cp, hw):
    x = wl.normal_f32(93, 0, (3, *hw, 270))
    g = cp.cprune_global_avgpool(cp.cprune_cast_input(_dev(x)), 270).float().cpu().numpy()
    ref = oracle.gap(oracle.round_bf16(x))
    scale = np.abs(oracle.round_bf16(x)).mean(axis=(1, 2))
    # one rounding to bf16 (8 significant bits: half a unit is at most 2^-8 of the value), float32 sums of at most 272 values
    assert np.all(np.abs(g[:, :270] - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -18 * scale) and np.all(g[:, 270:] == 0)


def block_tensors(seed, N, C_in, H, W, hidden, C_out):
    x = wl.normal_f32(seed, 0, (N, H, W, C_in))
    we = wl.normal_f32(seed, 1, (hidden, C_in, 1, 1), np.sqrt(2.0 / C_in))
    wd = wl.normal_f32(seed, 2, (hidden, 1, 3, 3), np.sqrt(2.0 / 9))
    wp = wl.normal_f32(seed, 3, (C_out, hidden, 1, 1), np.sqrt(2.0 / hidden))
    be, bd, bp = (wl.normal_f32(seed, 4 + j, (n,), 0.05) for j, n in enumerate((hidden, hidden, C_out)))
    return x, we, be, wd, bd, wp, bp


def block_reference(t, act, act_out, residual, matched):
    """The block as the chain of its three tasks in the oracle; matched: bf16 where the device rounds to bf16."""
    x, we, be, wd, bd, wp, bp = t
    rnd = oracle.round_bf16 if matched else (lambda a: np.asarray(a, dtype=np.float64))
    xr = rnd(x)
    h1 = rnd(oracle.conv2d(xr, rnd(we), be, 1, 0, 1, act))
    h2 = rnd(oracle.conv2d(h1, rnd(wd), bd, 1, 1, wd.shape[0], act))
    return oracle.conv2d(h2, rnd(wp), bp, 1, 0, 1, act_out, xr if residual else None, with_bound=True)


@pytest.mark.parametrize("case", [
    # N, C_in, H, W, hidden, C_out, act, residual: the stride-1 blocks of pruned MobileNetV2 at 14x14 and 7x7, then ragged
    # extents, channel counts off the 8 / 16 / 64 grid, one and several 64-channel chunks, relu (MnasNet) and no activation
    (3, 64, 14, 14, 288, 64, "relu6", True), (2, 64, 14, 14, 288, 96, "relu6", False), (2, 96, 14, 14, 432, 96, "relu6", True),
    (4, 160, 7, 7, 720, 160, "relu6", True), (2, 24, 9, 11, 100, 40, "relu", False), (1, 75, 13, 14, 75, 75, "none", True),
    (5, 8, 5, 4, 30, 12, "relu6", False), (2, 130, 12, 12, 64, 130, "relu", True), (1, 40, 7, 7, 200, 250, "relu", False)])
def test_fused_inverted_residual_block(cp, case):
    N, C_in, H, W, hidden, C_out, act, residual = case
    t = block_tensors(61, N, C_in, H, W, hidden, C_out)
    x, we, be, wd, bd, wp, bp = t
    blk = cp.cprune_block_plan(N, C_in, H, W, hidden, C_out, act, "none", residual)
    wq, bq = cp.cprune_block_pack(blk, _dev(we.reshape(hidden, C_in)), _dev(be), _dev(wd.reshape(hidden, 9)), _dev(bd),
                                  _dev(wp.reshape(C_out, hidden)), _dev(bp))
    y = cp.cprune_block_run(blk, cp.cprune_cast_input(_dev(x)), wq, bq).float().cpu().numpy()
    cp.cprune_poll_device_status()
    assert y.shape == (N, H, W, blk.k_pad) and np.all(y[..., C_out:] == 0)
    ref, bound = block_reference(t, act, "none", residual, matched=False)
    ref_m, bound_m = block_reference(t, act, "none", residual, matched=True)
    got = y[..., :C_out]
    r1 = float(np.max(np.abs(got - ref) / bound))
    # against the matched chain: the stored result's own rounding, plus what a differently rounded hidden value (float32
    # against float64 sums under the two bf16 roundings inside the block) can move: far below 1e-3 of the scale
    r2 = float(np.max(np.abs(got - ref_m) / (MATCH_REL * np.abs(ref_m) + 1e-3 * bound_m)))
    WORST["fused block %s" % (case,)] = (r1, r2)
    assert r1 <= TOL and r2 <= 1.0, (case, r1, r2)
    # the same three tasks run separately give the same values up to those rounding flips
    p1 = cp.cprune_task_plan(N, C_in, H, W, hidden, 1, 1, 1, 0, 1, act)
    p2 = cp.cprune_task_plan(N, hidden, H, W, hidden, 3, 3, 1, 1, hidden, act)
    p3 = cp.cprune_task_plan(N, hidden, H, W, C_out, 1, 1, 1, 0, 1, "none", residual)
    xb = cp.cprune_cast_input(_dev(x))
    a = cp.cprune_task_run(p1, xb, *cp.cprune_pack_weights(p1, _dev(we), _dev(be)))
    b = cp.cprune_task_run(p2, a, *cp.cprune_pack_weights(p2, _dev(wd), _dev(bd)))
    c = cp.cprune_task_run(p3, b, *cp.cprune_pack_weights(p3, _dev(wp), _dev(bp)), xb if residual else None)
    sep = c.float().cpu().numpy()[..., :C_out]
    assert np.max(np.abs(sep - got) / (MATCH_REL * np.abs(ref_m) + 1e-3 * bound_m)) <= 2.0


@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, act, res: one and two pixel blocks per tile, several tiles per thread block, rows and columns beyond the image,
    # an odd number of 8-channel groups, two chunks of channels, more than 64 and more than 256 filters (two MMAs), a residual
    (64, 32, 57, 55, 16, 3, "relu6", False), (40, 40, 21, 23, 40, 3, "relu", True), (70, 200, 14, 14, 72, 3, "relu6", False),
    (150, 296, 9, 11, 100, 3, "none", False), (80, 72, 28, 28, 320, 5, "relu", False), (64, 144, 13, 13, 144, 5, "none", True),
    (3, 24, 56, 56, 20, 3, "relu", False)])
def test_depthwise_and_1x1_tasks_as_one_kernel(cp, case):
    N, C, H, W, K, R, act, res = case
    x, w, b, _ = wl.conv_task_tensors(110, N, C, H, W, C, R, R, C)
    _, w2, b2, _ = wl.conv_task_tensors(111, 1, C, 1, 1, K, 1, 1)
    dw = cp.cprune_task_plan(N, C, H, W, C, R, R, 1, R // 2, C, act)
    pj = cp.cprune_task_plan(N, C, H, W, K, 1, 1, 1, 0, 1, act, res)
    p1, p2, fc = cp.cprune_pack_weights(dw, _dev(w), _dev(b)), cp.cprune_pack_weights(pj, _dev(w2), _dev(b2)), cp.cprune_fc_pack(torch.ones((8, K), device="cuda"))
    def build(flag):
        tasks = [cp.TaskDesc(op=cp.OP_CONV, in_=0, out=1, res=-1, plan=dw.handle, w=p1[0].data_ptr(), b=p1[1].data_ptr(), p0=flag),
                 cp.TaskDesc(op=cp.OP_CONV, in_=1, out=2, res=0 if res else -1, plan=pj.handle, w=p2[0].data_ptr(), b=p2[1].data_ptr()),
                 cp.TaskDesc(op=cp.OP_GAP, in_=2, out=3, res=-1),
                 cp.TaskDesc(op=cp.OP_FC, in_=3, out=4, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=K, p1=8)]
        return cp.cprune_model_create(N, H, W, C, tasks, keep_alive=(dw, pj, p1, p2, fc))
    model, plain = build(cp.CONV_WITH_NEXT), build(0)
    assert model.launches == plain.launches - 1
    for use_graph in (False, True):
        cp.cprune_model_run(model, _dev(x), use_graph=use_graph)
    cp.cprune_model_run(plain, _dev(x))
    y = model.copy_tensor(2).float().cpu().numpy()
    cp.cprune_poll_device_status()
    # the tensor in between is not stored, but can be had; the second product against the oracle on these very values
    h = model.copy_tensor(1)
    assert torch.equal(h, plain.copy_tensor(1))
    h, rb = h.float().cpu().numpy()[..., :C], oracle.round_bf16
    r = rb(x) if res else None
    ref, bound = oracle.conv2d(h, w2, b2, 1, 0, 1, act, r, with_bound=True)
    ref_m, bound_m = oracle.conv2d(h, rb(w2), b2, 1, 0, 1, act, r, with_bound=True)
    assert np.all(y[..., K:] == 0)
    check_values("pair %s" % (case,), y[..., :K], ref, bound, ref_m, bound_m)
    # a pixel that is no number reaches only the outputs whose window holds it
    bad = x.copy()
    bad[N - 1, 4, 3, 5] = np.nan
    cp.cprune_model_run(model, _dev(bad))
    cp.cprune_model_run(plain, _dev(bad))
    z, want = model.copy_tensor(2).float().cpu().numpy(), plain.copy_tensor(2).float().cpu().numpy()
    cp.cprune_poll_device_status()
    lo, hi = 4 - R // 2, 4 + R // 2 + 1
    out = np.ones(y.shape[:3], dtype=bool)
    out[N - 1, max(0, lo):hi, max(0, lo - 1):hi - 1] = False
    assert np.array_equal(z[out], y[out]) and np.array_equal(np.isnan(z), np.isnan(want))
    # an address handed out is kept up to date from then on: the tasks run separately
    cp.cprune_model_run(model, _dev(x), use_graph=True)
    model.tensor(1)
    assert model.launches == plain.launches
    cp.cprune_model_run(model, _dev(x), use_graph=True)
    cp.cprune_model_run(plain, _dev(x))
    assert torch.equal(model.copy_tensor(2), plain.copy_tensor(2))


def test_pairs_are_an_option_of_their_own(cp):
    from paper_2207_01260_b200.pipeline import PrunedNetwork
    table = wl.mobilenet_v2()
    table["input"] = (96, 96, 3)
    weights, x = wl.model_weights(table), _dev(wl.normal_f32(120, 0, (20, 96, 96, 3)))
    nets = {kw: PrunedNetwork(table, weights, 20, **dict(kw)) for kw in ((), (("fuse_blocks", False),), (("fuse_blocks", False), ("fuse_pairs", True)), (("fuse_pairs", False),))}
    auto, separate, pairs, off = nets.values()
    assert auto.model.launches == pairs.model.launches < separate.model.launches == off.model.launches
    assert torch.equal(pairs.run(x), auto.run(x)) and torch.equal(off.run(x), separate.run(x))
    ref = separate.run(x)
    assert torch.linalg.vector_norm(pairs.run(x) - ref) <= 1e-2 * torch.linalg.vector_norm(ref)
    cp.cprune_poll_device_status()


def test_the_address_of_a_tensor_between_two_tasks_beside_passes_of_another_thread(cp):
    import threading
    N, C, H, K = 32, 48, 28, 24
    x, w, b, _ = wl.conv_task_tensors(118, N, C, H, H, C, 3, 3, C)
    _, w2, b2, _ = wl.conv_task_tensors(119, 1, C, 1, 1, K, 1, 1)
    dw, pj = cp.cprune_task_plan(N, C, H, H, C, 3, 3, 1, 1, C), cp.cprune_task_plan(N, C, H, H, K, 1, 1, 1, 0)
    p1, p2, fc = cp.cprune_pack_weights(dw, _dev(w), _dev(b)), cp.cprune_pack_weights(pj, _dev(w2), _dev(b2)), cp.cprune_fc_pack(torch.ones((8, K), device="cuda"))

    def build():
        tasks = [cp.TaskDesc(op=cp.OP_CONV, in_=0, out=1, res=-1, plan=dw.handle, w=p1[0].data_ptr(), b=p1[1].data_ptr(), p0=cp.CONV_WITH_NEXT),
                 cp.TaskDesc(op=cp.OP_CONV, in_=1, out=2, res=-1, plan=pj.handle, w=p2[0].data_ptr(), b=p2[1].data_ptr()),
                 cp.TaskDesc(op=cp.OP_GAP, in_=2, out=3, res=-1),
                 cp.TaskDesc(op=cp.OP_FC, in_=3, out=4, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=K, p1=8)]
        return cp.cprune_model_create(N, H, H, C, tasks, keep_alive=(dw, pj, p1, p2, fc))

    xd, logits = _dev(x), torch.zeros((N, 8), device="cuda")
    model = build()
    one = model.launches
    model.tensor(1)                                   # before any pass
    assert model.launches == one + 1
    cp.cprune_model_run(model, xd, logits)
    h, y, want = model.copy_tensor(1), model.copy_tensor(2), logits.clone()
    for use_graph in (False, True):
        model, errors, started = build(), [], threading.Event()

        def passes():
            try:
                stream = torch.cuda.Stream()
                with torch.cuda.stream(stream):
                    for i in range(60):
                        cp.cprune_model_run(model, xd, logits, use_graph=use_graph)
                        if i == 10:
                            started.set()
                stream.synchronize()
            except Exception as e:                    # noqa: BLE001
                errors.append(e)
                started.set()

        t = threading.Thread(target=passes)
        t.start()
        started.wait(60)
        model.tensor(1)
        t.join(60)
        assert not errors and not t.is_alive()
        torch.cuda.synchronize()
        assert model.launches == one + 1 and torch.equal(model.copy_tensor(1), h)
        # (one kernel or two, as the last pass had it: bf16 results that may be rounded the other way)
        assert torch.allclose(model.copy_tensor(2).float(), y.float(), rtol=2.0 ** -7, atol=1e-3)
        assert torch.allclose(logits, want, rtol=1e-2, atol=1e-3 * float(want.abs().max()) + 1e-3)
    cp.cprune_poll_device_status()


@pytest.mark.parametrize("case", [
    # N, C, H, K, R, act, res: more than 256 filters, whose two MMAs are wider than the stored pixel; one tile and several per thread block
    (1, 32, 56, 257, 5, "relu", False), (64, 72, 14, 272, 3, "none", False), (64, 72, 14, 260, 3, "none", True), (64, 32, 28, 300, 5, "relu6", False),
    (90, 32, 16, 304, 3, "relu", True)])
def test_depthwise_and_wide_1x1_tasks_as_one_kernel_stay_in_their_pixels(cp, case):
    N, C, H, K, R, act, res = case
    x, w, b, _ = wl.conv_task_tensors(112, N, C, H, H, C, R, R, C)
    _, w2, b2, _ = wl.conv_task_tensors(113, 1, C, 1, 1, K, 1, 1)
    _, w3, b3, _ = wl.conv_task_tensors(114, 1, C, 1, 1, K, 1, 1)
    dw = cp.cprune_task_plan(N, C, H, H, C, R, R, 1, R // 2, C, act)
    pj = cp.cprune_task_plan(N, C, H, H, K, 1, 1, 1, 0, 1, act, res)
    side = cp.cprune_task_plan(N, C, H, H, K, 1, 1, 1, 0, 1, "none")
    p1, p2, p3 = (cp.cprune_pack_weights(*t) for t in ((dw, _dev(w), _dev(b)), (pj, _dev(w2), _dev(b2)), (side, _dev(w3), _dev(b3))))
    fc = cp.cprune_fc_pack(torch.ones((8, K), device="cuda"))

    def build(flag):
        # tensors lie in memory in the order of their ids: behind the pair's result (3) comes a copy of the image (4), its input
        conv = lambda i, o, plan, p, r=-1, f=0: cp.TaskDesc(op=cp.OP_CONV, in_=i, out=o, res=r, plan=plan.handle, w=p[0].data_ptr(), b=p[1].data_ptr(), p0=f)
        tasks = [cp.TaskDesc(op=cp.OP_MAXPOOL, in_=0, out=4, res=-1, p0=1, p1=1), conv(4, 6, side, p3), conv(4, 5, dw, p1, f=flag),
                 conv(5, 3, pj, p2, 6 if res else -1), cp.TaskDesc(op=cp.OP_GAP, in_=3, out=7, res=-1),
                 cp.TaskDesc(op=cp.OP_FC, in_=7, out=8, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=K, p1=8)]
        return cp.cprune_model_create(N, H, H, C, tasks, keep_alive=(dw, pj, side, p1, p2, p3, fc))

    model, plain = build(cp.CONV_WITH_NEXT), build(0)
    assert model.launches == plain.launches - 1
    for m in (model, plain):
        for _ in range(2):
            cp.cprune_model_run(m, _dev(x))
    y, want = model.copy_tensor(3).float().cpu().numpy(), plain.copy_tensor(3).float().cpu().numpy()
    h = model.copy_tensor(5).float().cpu().numpy()[..., :C]
    assert torch.equal(model.copy_tensor(4), plain.copy_tensor(4)) and torch.equal(model.copy_tensor(6), plain.copy_tensor(6))
    r = plain.copy_tensor(6).float().cpu().numpy()[..., :K] if res else None
    cp.cprune_poll_device_status()
    assert np.all(y[..., K:] == 0)
    ref, bound = oracle.conv2d(h, w2, b2, 1, 0, 1, act, r, with_bound=True)
    ref_m, bound_m = oracle.conv2d(h, oracle.round_bf16(w2), b2, 1, 0, 1, act, r, with_bound=True)
    check_values("wide pair %s" % (case,), y[..., :K], ref, bound, ref_m, bound_m)
    check_values("wide pair, separate %s" % (case,), want[..., :K], ref, bound, ref_m, bound_m)


@pytest.mark.parametrize("which,offset", [(0, 4), (0, 8), (1, 4), (2, 1), (3, 2)])
def test_a_pair_refuses_the_parameters_that_its_tasks_refuse(cp, which, offset):
    # 0, 1: depthwise and 1x1 filters off a 16-byte boundary; 2, 3: their biases off a 4-byte one.  The host refuses: no kernel reads them
    N, C, H, K = 64, 32, 28, 16
    _, w, b, _ = wl.conv_task_tensors(115, 1, C, H, H, C, 3, 3, C)
    _, w2, b2, _ = wl.conv_task_tensors(116, 1, C, 1, 1, K, 1, 1)
    dw, pj = cp.cprune_task_plan(N, C, H, H, C, 3, 3, 1, 1, C, "relu"), cp.cprune_task_plan(N, C, H, H, K, 1, 1, 1, 0)
    packed = [cp.cprune_pack_weights(dw, _dev(w), _dev(b)), cp.cprune_pack_weights(pj, _dev(w2), _dev(b2))]
    bytes_ = [t.contiguous().view(torch.uint8).reshape(-1) for t in (packed[0][0], packed[1][0], packed[0][1], packed[1][1])]
    moved = torch.empty(bytes_[which].numel() + 16, dtype=torch.uint8, device="cuda")
    moved[offset:offset + bytes_[which].numel()] = bytes_[which]
    ptr = [t.data_ptr() for t in bytes_]
    fc = cp.cprune_fc_pack(torch.ones((8, K), device="cuda"))

    def build(p):
        tasks = [cp.TaskDesc(op=cp.OP_CONV, in_=0, out=1, res=-1, plan=dw.handle, w=p[0], b=p[2], p0=cp.CONV_WITH_NEXT),
                 cp.TaskDesc(op=cp.OP_CONV, in_=1, out=2, res=-1, plan=pj.handle, w=p[1], b=p[3]),
                 cp.TaskDesc(op=cp.OP_GAP, in_=2, out=3, res=-1),
                 cp.TaskDesc(op=cp.OP_FC, in_=3, out=4, res=-1, w=fc[0].data_ptr(), b=fc[1].data_ptr(), p0=K, p1=8)]
        return cp.cprune_model_create(N, H, H, C, tasks, keep_alive=(dw, pj, packed, moved, fc))

    good = build(ptr)
    ptr[which] = moved.data_ptr() + offset
    bad = build(ptr)
    x = _dev(wl.normal_f32(117, 0, (N, H, H, C)))
    for use_graph in (False, True):
        with pytest.raises(cp.CpruneError) as e:
            cp.cprune_model_run(bad, x, use_graph=use_graph)
        assert e.value.status == 1                    # CPRUNE_ERR_INVALID_ARG
    assert bad.launches == good.launches + 1
    cp.cprune_model_run(good, x)
    cp.cprune_poll_device_status()


def test_mobilenet_v2_with_and_without_pairs(cp):
    from paper_2207_01260_b200.pipeline import PrunedNetwork
    table = wl.mobilenet_v2()
    weights = wl.model_weights(table)
    x = wl.model_input(table, 1)
    pairs, plain = PrunedNetwork(table, weights, 1), PrunedNetwork(table, weights, 1, fuse_blocks=False)
    assert pairs.model.launches < plain.model.launches
    a, b = pairs.run(_dev(x)).cpu().numpy(), plain.run(_dev(x)).cpu().numpy()
    cp.cprune_poll_device_status()
    assert np.linalg.norm(a - b) <= 1e-2 * np.linalg.norm(b)           # the order of the float32 sums differs, at batch 1 in 4 of 17 blocks
    pw, _ = oracle.prune_model(table, weights)
    ref = oracle.model_ref(table, pw, x, matched=True)
    assert np.linalg.norm(a - ref) <= 1e-2 * np.linalg.norm(ref)
    for name in ("b1_dw", "b3_dw", "b9_dw"):                           # depthwise results can be had whether stored or not
        out = wl.layer_by_name(table)[name]["out"]
        u, v = pairs.activation(out), plain.activation(out)
        assert np.linalg.norm(u - v) <= 1e-2 * np.linalg.norm(v)


def test_fused_block_argument_errors_and_unsupported_shapes(cp):
    for args in ((2, 64, 28, 28, 288, 64), (2, 256, 14, 14, 512, 64), (2, 64, 14, 14, 288, 320)):   # image too large, C_in, C_out
        with pytest.raises(cp.CpruneError) as e:
            cp.cprune_block_plan(*args)
        assert e.value.status == 2
    with pytest.raises(cp.CpruneError) as e:
        cp.cprune_block_plan(2, 64, 14, 14, 288, 96, residual=True)        # a residual needs C_in == C_out
    assert e.value.status == 1
    a = cp.cprune_block_plan(2, 64, 14, 14, 288, 64, residual=True)
    b = cp.cprune_block_plan(2, 64, 14, 14, 288, 64, residual=True)
    assert a.handle.value == b.handle.value and a.unfused_bytes > 2 * a.algorithmic_bytes


def test_mobilenet_v2_with_and_without_fused_blocks(cp):
    from paper_2207_01260_b200.pipeline import PrunedNetwork
    table = wl.mobilenet_v2()
    weights = wl.model_weights(table)
    x = wl.model_input(table, 4)
    fused = PrunedNetwork(table, weights, 4, fuse_blocks=True)
    plain = PrunedNetwork(table, weights, 4, fuse_blocks=False)
    # the stride-1 blocks of the 14x14 and 7x7 stages, except the last one (320 filters do not fit one image's accumulator)
    assert sorted(fused.blocks) == sorted(["b8_exp", "b9_exp", "b10_exp", "b11_exp", "b12_exp", "b13_exp", "b15_exp", "b16_exp"])
    assert not PrunedNetwork(table, weights, 64).blocks and PrunedNetwork(table, weights, 2).blocks      # the default follows the batch
    assert fused.model.launches == plain.model.launches - sum(3 - (2 if b.splits > 1 else 1) for b in fused.blocks.values())
    a = fused.run(_dev(x)).cpu().numpy()
    b = plain.run(_dev(x)).cpu().numpy()
    cp.cprune_poll_device_status()
    assert np.linalg.norm(a - b) <= 3e-3 * np.linalg.norm(b)
    pw, _ = oracle.prune_model(table, weights)
    ref = oracle.model_ref(table, pw, x, matched=True)
    assert np.linalg.norm(a - ref) <= 1e-2 * np.linalg.norm(ref)
    print("\nfused blocks: %s; launches %d -> %d" % (sorted(fused.blocks), plain.model.launches, fused.model.launches))


def test_shared_selection_and_shortcut_pruned_resnet(cp):
    # dependency-aware pruning: one ranking for the layers whose outputs meet in a residual add
    ws = [wl.normal_f32(51, 1, (96, 20, 3, 3), 0.1), wl.normal_f32(51, 2, (96, 64, 1, 1), 0.1), wl.normal_f32(51, 3, (96, 7, 3, 3), 0.1)]
    ws[0][5] = ws[0][4]
    ws[1][5] = ws[1][4]
    ws[2][5] = -ws[2][4]                   # filters 4 and 5 tie exactly across the group: the lower index wins
    for keep in (1, 5, 48, 95, 96):
        kept = cp.cprune_select_shared([_dev(w) for w in ws], keep)
        assert np.array_equal(kept.cpu().numpy(), oracle.select_indices_shared(ws, keep)), keep
    cp.cprune_poll_device_status()
    one = cp.cprune_select_shared([_dev(ws[0])], 40)
    assert np.array_equal(one.cpu().numpy(), oracle.select_indices(ws[0], 40))
    net, _, _ = model_parity(cp, "resnet18_shared", 2, hw=64)
    assert net.plans["l2b1_conv2"].K == 96 and net.plans["l2b2_conv1"].C == 96 and net.plans["stem"].K == 48


def test_intermediate_activations_match(cp):
    from paper_2207_01260_b200.pipeline import PrunedNetwork
    table = wl.resnet18()
    table["input"] = (64, 64, 3)
    weights = wl.model_weights(table)
    x = wl.model_input(table, 2)
    net = PrunedNetwork(table, weights, 2)
    net.run(_dev(x))
    pw, _ = oracle.prune_model(table, weights)
    _, tensors = oracle.model_ref(table, pw, x, matched=True, keep_tensors=True)
    # the stem's 3x3 max-pool is fused into the stem task: its unpooled output "s0" is never stored
    for name in ("p0", "l1b1_h", "l1b1_o", "l2b1_id", "l2b1_o", "l4b2_o", "g"):
        got = net.activation(name)
        ref = tensors[name].reshape(got.shape)
        rel = np.linalg.norm(got - ref) / np.linalg.norm(ref)
        assert rel <= 1e-2, (name, rel)
    net = PrunedNetwork(table, weights, 2, fuse_pool=False)
    net.run(_dev(x))
    for name in ("s0", "p0"):
        got = net.activation(name)
        ref = tensors[name].reshape(got.shape)
        rel = np.linalg.norm(got - ref) / np.linalg.norm(ref)
        assert rel <= 1e-2, (name, rel)


@pytest.mark.parametrize("act", ["none", "relu", "relu6"])
@pytest.mark.parametrize("case", [
    # N, C, H, K, R, stride, groups, variant: the patch kernel with resident filters, with a ring of filter rows and of taps, on whole
    # images, on flat tasks staged by 64 filters and as they lie in memory; im2col in both orientations; depthwise
    (64, 64, 28, 48, 3, 1, 1, 1), (64, 256, 14, 89, 3, 1, 1, 1), (64, 256, 14, 256, 3, 1, 1, 1), (128, 96, 8, 80, 3, 1, 1, 1),
    (64, 32, 28, 200, 1, 1, 1, 1), (64, 48, 56, 72, 1, 1, 1, 2), (64, 64, 28, 96, 3, 2, 1, 0), (64, 64, 28, 200, 3, 2, 1, 0),
    (4, 40, 14, 40, 3, 1, 40, 0),
    # few pixels
    (2, 64, 16, 48, 3, 1, 1, 3), (2, 64, 16, 48, 1, 1, 1, 3), (2, 64, 16, 200, 3, 2, 1, 3)])
def test_a_nan_pixel_reaches_only_the_outputs_whose_window_holds_it(cp, case, act):
    # every kernel answers alike: NaN without an activation, 0 under the clamps (the clamp returns the operand that is a number)
    N, C, H, K, R, stride, groups, variant = case
    plan = cp.cprune_task_plan(N, C, H, H, K, R, R, stride, R // 2, groups, act)
    assert plan.variant == variant
    x, w, b, _ = wl.conv_task_tensors(97, N, C, H, H, K, R, R, groups)
    wp, bp = cp.cprune_pack_weights(plan, _dev(w), _dev(b))
    clean = cp.cprune_cast_input(_dev(x))
    bad, h, v, c = clean.clone(), 4, 5, 3
    bad[1, h, v, c] = float("nan")
    a, y = (cp.cprune_task_run(plan, t, wp, bp).clone()[..., :K].float() for t in (clean, bad))
    cp.cprune_poll_device_status()
    touched = torch.zeros_like(a, dtype=torch.bool)
    p = torch.arange(plan.P, device="cuda") * stride - R // 2
    rows, cols = (p <= h) & (h < p + R), (p <= v) & (v < p + R)
    touched[1] = (rows[:, None] & cols[None, :])[..., None] & (torch.ones(K, dtype=torch.bool, device="cuda") if groups == 1 else torch.arange(K, device="cuda") == c)
    assert torch.equal(y[~touched], a[~touched])
    got = y[touched]
    assert torch.isnan(got).all() if act == "none" else (got == 0).all()


def test_a_nan_in_a_pooled_window_of_few_pixels(cp):
    # a maximum skips a NaN beside numbers and is a NaN when the whole window is (as the separate pooling pass has it)
    N, C, H, K = 2, 64, 8, 48
    x, w, b, _ = wl.conv_task_tensors(98, N, C, H, H, K, 1, 1)
    x[0, 2, 2, 0] = np.nan                        # one pixel of the pooled pixel (1, 1)
    x[1, 4:6, 6:8, 5] = np.nan                    # all four of (2, 3)
    plan = cp.cprune_task_plan(N, C, H, H, K, 1, 1, 1, 0, 1, "none", False, "max2x2")
    assert plan.variant == 3
    y = cp.cprune_task_run(plan, cp.cprune_cast_input(_dev(x)), *cp.cprune_pack_weights(plan, _dev(w), _dev(b))).float()[..., :K]
    assert torch.isnan(y).nonzero()[:, :3].unique(dim=0).tolist() == [[1, 2, 3]] and torch.isnan(y[1, 2, 3]).all()
    assert torch.isfinite(y[0]).all()


@pytest.mark.parametrize("case", [
    # N, C, H, K, R, stride, groups: depthwise 3x3 and 5x5, the patch kernel (bias in shared memory; staged as in memory), filters
    # on the row side of the im2col kernel, few pixels
    (4, 40, 14, 40, 3, 1, 40), (4, 40, 14, 40, 5, 2, 40), (64, 64, 28, 48, 3, 1, 1), (64, 48, 56, 72, 1, 1, 1), (64, 64, 28, 96, 3, 2, 1),
    (2, 64, 16, 48, 3, 1, 1)])
def test_a_packed_bias_at_any_float_address(cp, case):
    N, C, H, K, R, stride, groups = case
    plan = cp.cprune_task_plan(N, C, H, H, K, R, R, stride, R // 2, groups)
    x, w, b, _ = wl.conv_task_tensors(100, N, C, H, H, K, R, R, groups)
    xb, (wp, bp) = cp.cprune_cast_input(_dev(x)), cp.cprune_pack_weights(plan, _dev(w), _dev(b))
    y = cp.cprune_task_run(plan, xb, wp, bp)
    for off in (1, 2, 3):
        moved = torch.empty(bp.numel() + off, device="cuda")[off:]
        moved.copy_(bp)
        assert torch.equal(cp.cprune_task_run(plan, xb, wp, moved), y)
    cp.cprune_poll_device_status()


@pytest.mark.parametrize("raw", [True, False])
def test_calls_go_to_the_current_stream(cp, raw, monkeypatch):
    # with torch's call for the raw handle, which it does not promise, and without
    from paper_2207_01260_b200 import binding
    if not raw:
        monkeypatch.setattr(binding, "_raw_stream", None)
    s = torch.cuda.Stream()
    assert binding._stream() == torch.cuda.current_stream().cuda_stream and binding._stream(s) == s.cuda_stream
    with torch.cuda.stream(s):
        assert binding._stream() == s.cuda_stream


def test_plan_cache_shares_repeated_shapes(cp):
    from paper_2207_01260_b200.pipeline import PrunedNetwork
    table = wl.resnet18()
    net = PrunedNetwork(table, wl.model_weights(table), 1)
    handles = {p.handle.value for p in net.plans.values()}
    assert len(net.plans) == 20 and len(handles) == 15          # 20 conv tasks, 15 distinct shapes
