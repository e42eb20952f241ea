"""GPU parity: the CUDA library, called through its C ABI, against the CPU oracle on the same
seeded inputs. Sample streams bit-exact; models within relative L2 error 1e-4 (logistic, squared)
or 1e-3 (hinge: a margin within rounding of 1 may flip one subgradient)."""
import numpy as np
import pytest
import torch

import oracle
import wpsgd_inputs as wi

pytestmark = pytest.mark.gpu

HINGE, LOGISTIC, SQUARED = 0, 1, 2
TOL = {HINGE: 1e-3, LOGISTIC: 1e-4, SQUARED: 1e-4}


@pytest.fixture(scope="module")
def P(wpsgd_lib):
    import paper_1708_04801_b200 as pkg

    return pkg


def rel_l2(a, b):
    a = np.asarray(a, dtype=np.float64)
    b = np.asarray(b, dtype=np.float64)
    den = np.linalg.norm(b)
    return float(np.linalg.norm(a - b) / den) if den > 0 else float(np.linalg.norm(a))


def gpu_solve(P, wl_cpu, options=None, r=0.0):
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        for k_, v_ in (options or {}).items():
            ctx.set_option(k_, v_)
        ctx.run_workload(wl)
        v = ctx.combine(r)
        W = ctx.get_models()
        wts, flag = ctx.get_weights(r)
        ctx.check()
        return v.cpu().numpy(), W.cpu().numpy(), wts, flag


def assert_parity(P, wl, options=None, r=0.0, tol=None):
    v, W, wts, flag = gpu_solve(P, wl, options, r)
    ov, oW, owts = oracle.solve(wl, r)
    tol = tol or TOL[wl.loss]
    np.testing.assert_allclose(wts, owts, rtol=1e-12)
    worst = max(rel_l2(W[j], oW[j]) for j in range(wl.k) if np.linalg.norm(oW[j]) > 0)
    assert worst <= tol, f"per-node model error {worst:.3e} > {tol}"
    err = rel_l2(v, ov)
    assert err <= tol, f"combined model error {err:.3e} > {tol}"
    return err


# ---- sample stream ------------------------------------------------------------------------------------
@pytest.mark.parametrize("seed,node,m,n_begin,count", [
    (0, 0, 4096, 0, 1000), (0, 3, 4096, 0, 250), (1, 15, 8192, 0, 20001), (7, 2, 1, 0, 17),
    (0xFFFFFFFFFFFFFFFF, 1023, (1 << 32) - 1, 0, 4099), (5, 9, 65536, 1, 1), (5, 9, 65536, 2, 3), (5, 9, 65536, 3, 6),
    (5, 9, 65536, 1237, 3763), (0x123456789ABCDEF1, 77, 2047, 999999999, 1025), (3, 1, 10, 0, 0),
    (2, 4, 3, (1 << 34) + 1, 13),
])
def test_sample_stream_bit_exact(P, seed, node, m, n_begin, count):
    with P.Context(2, 8) as ctx:
        got = ctx.sample_indices(seed, node, m, n_begin, count).cpu().numpy().view(np.uint32)
        ctx.check()
    want = oracle.sample_indices(seed, node, m, n_begin, count)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("seed,node,m,n_begin,count", [
    (0, 0, 4096, 0, 9000), (3, 7, 1, 0, 5), (3, 7, 2, 1, 9), (9, 1023, 1000, 998, 1005), (5, 2, 65537, 0, 70000),
    (0xFFFFFFFFFFFFFFFF, 4, (1 << 32) - 1, (1 << 33) + 3, 257), (1, 1, 5, 0, 0),
])
def test_shuffled_sample_stream_bit_exact(P, seed, node, m, n_begin, count):
    oracle.set_sampling(1)
    try:
        want = oracle.sample_indices(seed, node, m, n_begin, count)
    finally:
        oracle.set_sampling(0)
    with P.Context(2, 8) as ctx:
        ctx.set_option("sampling", 1)
        got = ctx.sample_indices(seed, node, m, n_begin, count).cpu().numpy().view(np.uint32)
        ctx.check()
    assert np.array_equal(got, want)


@pytest.mark.parametrize("cfg", [1, 2, 3, 4, 5])
def test_small_workloads_shuffled_order(P, cfg):
    oracle.set_sampling(1)
    try:
        assert_parity(P, wi.small(cfg), {"sampling": 1})
    finally:
        oracle.set_sampling(0)


# ---- the five workloads, scaled down, default kernel choice ---------------------------------------------
@pytest.mark.parametrize("cfg", [1, 2, 3, 4, 5])
def test_small_workloads_default_kernels(P, cfg):
    assert_parity(P, wi.small(cfg))


# ---- every dense kernel variant ----------------------------------------------------------------------
@pytest.mark.parametrize("variant,threads,prefetch", [(1, 0, 0), (2, 0, 2), (2, 0, 4), (2, 0, 8), (2, 128, 4), (2, 64, 8),
                                                      (2, 32, 2), (3, 0, 2), (3, 0, 4), (3, 0, 8), (4, 0, 0)])
@pytest.mark.parametrize("bf16", [False, True])
def test_dense_variants(P, variant, threads, prefetch, bf16):
    # d = 480: 120 fp32 / 60 bf16 16-byte chunks: ragged against 32-lane and 128-thread tiles
    wl = wi.config2(k=5, d=480, m=96, base_steps=333)
    if bf16:
        wl.X = wl.X.to(torch.bfloat16)
    assert_parity(P, wl, {"dense_variant": variant, "threads": threads, "prefetch": prefetch})


@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
@pytest.mark.parametrize("sched", [0, 1])
@pytest.mark.parametrize("variant", [1, 2, 3, 4, 5])
def test_losses_and_schedules(P, loss, sched, variant):
    wl = wi.config1(k=3, d=64, m=128, n_steps=(300, 150, 40))
    wl.loss, wl.sched = loss, sched
    wl.eta0 = 0.05 if sched else 0.01
    if loss == SQUARED:
        wl.y = (wl.y * 0.5 + 0.1).contiguous()
    assert_parity(P, wl, {"dense_variant": variant})


def test_generic_kernel_handles_unaligned_shapes(P):
    # d = 67 (not a multiple of 4), row stride 71: the register and the aligned blocked kernels do not apply
    g = torch.Generator().manual_seed(3)
    k, d, ld, m = 3, 67, 71, 50
    Xp = torch.randn(k * m, ld, generator=g) / 8
    y = torch.sign(torch.randn(k * m, generator=g))
    off = np.arange(k + 1, dtype=np.int64) * m
    n = np.array([200, 77, 0], dtype=np.int64)
    oW = oracle.run_dense(Xp, y, off, n, d, 0.05, 0, 1e-2, LOGISTIC, 11)
    Xd = Xp.cuda()
    with P.Context(k, d) as ctx:
        ctx.run(Xd[:, :d], y.cuda(), off, n, 0.05, 0, 1e-2, LOGISTIC, 11)
        W = ctx.get_models().cpu().numpy()
        ctx.check()
        with pytest.raises(P.WpsgdError) as e:
            ctx.set_option("dense_variant", 2)
            ctx.run(Xd[:, :d], y.cuda(), off, n, 0.05, 0, 1e-2, LOGISTIC, 11)
        assert e.value.status_name == "UNSUPPORTED"
    for j in range(2):
        assert rel_l2(W[j], oW[j]) <= 1e-4
    assert np.all(W[2] == 0)


def test_large_d_falls_back_and_matches(P):
    wl = wi.config2(k=2, d=8200, m=16, base_steps=40)  # beyond the register kernels' reach (the default spreads a row over a cluster)
    assert_parity(P, wl)


# ---- rounding of the update: eta lambda far below 2^-24 of the model -----------------------------------------------------
@pytest.mark.parametrize("variant,d,bf16", [(0, 17, False), (0, 999, False), (0, 1001, True), (1, 67, False), (1, 256, True), (2, 256, False),
                                            (2, 1000, True), (3, 64, False)])
def test_small_decays_are_not_rounded_away(P, variant, d, bf16):
    # eta lambda from 1e-6 down to 1.6e-8: where w (1 - eta lambda) is rounded on its own in every step, its error has the same
    # sign step after step (4e-5 after these 4000 steps). One rounding of w per step, half a unit in the last place at most and
    # of either sign, leaves sqrt(4000) 2^-24 = 3.8e-6 at three times its standard deviation, twice that with the margins' sums.
    g = torch.Generator().manual_seed(4)
    k, m, n = 2, 512, 4000
    X = torch.randn(k * m, d, generator=g) / np.sqrt(d)
    if bf16:
        X = X.to(torch.bfloat16)
    y = (X.float() @ torch.randn(d, generator=g) + 0.1 * torch.randn(k * m, generator=g)).contiguous()
    off, steps = np.array([0, m, 2 * m], dtype=np.int64), np.array([n, n // 2], dtype=np.int64)
    oW = oracle.run_dense(X, y, off, steps, d, 0.01, 1, 1e-4, SQUARED, 7)
    with P.Context(k, d) as ctx:
        ctx.set_option("dense_variant", variant)
        ctx.run(X.cuda(), y.cuda(), off, steps, 0.01, 1, 1e-4, SQUARED, 7)
        W = ctx.get_models().cpu().numpy()
        ctx.check()
    for j in range(k):
        assert rel_l2(W[j], oW[j]) <= 8e-6


# ---- blocked kernels with the decaying step size eta0 / sqrt(n): per-block tables instead of powers of one factor -------
@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
@pytest.mark.parametrize("kind", ["block_fp32", "block_bf16", "warp", "mma8", "mma16", "f32x16"])
def test_blocked_kernels_decaying_step_size(P, kind, loss):
    d = {"block_fp32": 1024, "block_bf16": 1000, "warp": 256, "mma8": 2048, "mma16": 2048, "f32x16": 1024}[kind]
    wl = wi.config2(k=4, d=d, m=96, base_steps=333)
    wl.n_steps[3] = 0
    wl.loss, wl.sched, wl.eta0, wl.lam = loss, 1, 0.3, 0.05  # eta_n lambda from 1.5e-2 down: the factors differ step by step
    if loss == SQUARED:
        wl.y = (wl.y * 0.3).contiguous()
    wl.w0 = torch.full((d,), 0.05)
    if kind not in ("block_fp32", "warp", "f32x16"):
        wl.X = wl.X.to(torch.bfloat16)
    opts = {"block_fp32": {"dense_variant": 4}, "block_bf16": {"dense_variant": 4}, "warp": {"dense_variant": 5},
            "mma8": {"dense_variant": 8, "block_samples": 8, "cluster": 2},
            "mma16": {"dense_variant": 8, "block_samples": 16, "cluster": 2},
            "f32x16": {"dense_variant": 9, "cluster": 4}}[kind]
    assert_parity(P, wl, opts)


def test_decaying_step_size_continue_keeps_the_step_numbers(P):
    # a continued chain must take eta of its own step numbers (first + n), also inside the per-block tables
    wl_cpu = wi.config2(k=3, d=1024, m=64, base_steps=8)
    wl_cpu.n_steps = np.array([203, 101, 50], dtype=np.int64)
    wl_cpu.sched, wl_cpu.eta0, wl_cpu.lam = 1, 0.3, 0.05
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.run(wl.X, wl.y, wl.shard_off, np.array([50, 50, 50]), wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        ctx.continue_(wl.X, wl.y, wl.shard_off, np.array([153, 51, 0]))
        seg = ctx.get_models().cpu().numpy()
        ctx.check()
    oW = oracle.run_dense(wl_cpu.X, wl_cpu.y, wl.shard_off, wl_cpu.n_steps, wl.d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
    for j in range(wl.k):
        assert rel_l2(seg[j], oW[j]) <= 1e-4


# ---- blocked kernel: block boundaries, ring depths, column tilings ----------------------------------------
@pytest.mark.parametrize("n_steps", [(1, 7, 8), (9, 15, 16), (17, 0, 64), (333, 250, 3)])
@pytest.mark.parametrize("stages", [2, 3, 4])
def test_blocked_kernel_block_boundaries_and_ring_depths(P, n_steps, stages):
    wl = wi.config2(k=3, d=1024, m=64, base_steps=8)
    wl.n_steps = np.array(n_steps, dtype=np.int64)
    wl.w0 = torch.full((1024,), 0.1)
    assert_parity(P, wl, {"dense_variant": 4, "stages": stages})


@pytest.mark.parametrize("d,bf16", [(64, False), (480, False), (1024, False), (2048, False), (1536, False), (64, True),
                                     (1000, True), (4096, True), (3008, True)])
@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
def test_blocked_kernel_column_tilings(P, d, bf16, loss):
    wl = wi.config2(k=3, d=d, m=48, base_steps=210)
    wl.loss = loss
    if loss == SQUARED:
        wl.y = (wl.y * 0.3).contiguous()
    if bf16:
        wl.X = wl.X.to(torch.bfloat16)
    assert_parity(P, wl, {"dense_variant": 4})


@pytest.mark.parametrize("d,bf16", [(64, False), (200, False), (256, False), (8, False), (72, True), (512, True)])
@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
@pytest.mark.parametrize("stages", [2, 3])
def test_blocked_warp_kernel(P, d, bf16, loss, stages):
    # k = 11: three CTAs of four warps, the last one with an idle warp; step counts with ragged last blocks
    wl = wi.config5(k=11, d=d, m=40, total_steps=11 * 131, rho=6.0)
    wl.n_steps[3] = 0
    wl.n_steps[7] = 5
    wl.loss = loss
    if loss == SQUARED:
        wl.y = (wl.y * 0.3).contiguous()
    if bf16:
        wl.X = wl.X.to(torch.bfloat16)
    wl.w0 = torch.full((d,), 0.05)
    assert_parity(P, wl, {"dense_variant": 5, "stages": stages})


def test_blocked_warp_kernel_limits(P):
    wl = wi.config2(k=2, d=480, m=16, base_steps=20)  # 120 chunks: too wide for a warp
    with pytest.raises(P.WpsgdError) as e:
        gpu_solve(P, wl, {"dense_variant": 5})
    assert e.value.status_name == "UNSUPPORTED"


@pytest.mark.parametrize("d,bf16", [(1024, False), (2048, False), (4096, True)])
def test_bounded_wait_for_rows_reports_timeout_and_context_survives(P, d, bf16):
    # Failure detection without a fault: the rows of block 3 are never requested (test hook), so the bounded
    # wait for them runs out; the kernel flags it, leaves in step and returns, and the next run is clean.
    wl_cpu = wi.config2(k=3, d=d, m=32, base_steps=120)
    if bf16:
        wl_cpu.X = wl_cpu.X.to(torch.bfloat16)
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.set_option("dense_variant", 4)
        ctx.set_option("spin_limit", 2000)
        ctx.set_option("test_drop_block", 3)
        ctx.run_workload(wl)
        with pytest.raises(P.WpsgdError) as e:
            ctx.check()
        assert e.value.status_name == "TIMEOUT"
        ctx.set_option("test_drop_block", -1)
        ctx.set_option("spin_limit", 1 << 20)
        ctx.run_workload(wl)
        v = ctx.combine().cpu().numpy()
        ctx.check()
    ov, _, _ = oracle.solve(wl_cpu)
    assert rel_l2(v, ov) <= 1e-4


# ---- tensor-core cluster kernel (bf16 rows): Gram block and margins from mma, model split into three bf16 rows; blocks
# of 8 samples (every loss) or 16 samples (squared and hinge) -----------------------------------------------------------
MMA_BLOCKS = [8, 16]


def _mma(block, wl, **more):
    """Options that select the tensor-core kernel with the given block size."""
    return dict({"dense_variant": 8, "block_samples": block}, **more)


@pytest.mark.parametrize("cluster", [1, 2, 4])
@pytest.mark.parametrize("d", [480, 488, 8, 264])
@pytest.mark.parametrize("block", MMA_BLOCKS)
def test_mma_kernel_ragged_shapes(P, cluster, d, block):
    # 60 / 61 / 1 / 33 chunks of 8 columns: odd chunk counts leave half a 16-column tile empty, the last CTA of a
    # cluster owns a ragged slice, and with d = 8 only one CTA can exist
    if d == 8 and cluster > 1:
        pytest.skip("fewer chunks than CTAs")
    wl = wi.config2(k=5, d=d, m=96, base_steps=333)
    wl.n_steps[2] = 0
    wl.w0 = torch.full((d,), 0.05)
    wl.X = wl.X.to(torch.bfloat16)
    assert_parity(P, wl, _mma(block, wl, cluster=cluster))


@pytest.mark.parametrize("d,cluster", [(4096, 2), (4096, 4), (2048, 1), (4096, 8), (3008, 2), (1024, 8)])
@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
@pytest.mark.parametrize("block", MMA_BLOCKS)
def test_mma_kernel_losses_and_widths(P, d, cluster, loss, block):
    wl = wi.config2(k=3, d=d, m=48, base_steps=210)
    wl.loss = loss
    if loss == SQUARED:
        wl.y = (wl.y * 0.3).contiguous()
    wl.X = wl.X.to(torch.bfloat16)
    assert_parity(P, wl, _mma(block, wl, cluster=cluster))


@pytest.mark.parametrize("n_steps", [(1, 7, 8), (9, 15, 16), (17, 0, 64), (333, 250, 3), (31, 32, 33)])
@pytest.mark.parametrize("stages", [2, 3, 4])
@pytest.mark.parametrize("block", MMA_BLOCKS)
def test_mma_kernel_block_boundaries_and_ring_depths(P, n_steps, stages, block):
    wl = wi.config2(k=3, d=1024, m=64, base_steps=8)
    wl.n_steps = np.array(n_steps, dtype=np.int64)
    wl.w0 = torch.full((1024,), 0.1)
    wl.X = wl.X.to(torch.bfloat16)
    assert_parity(P, wl, _mma(block, wl, cluster=2, stages=stages))


@pytest.mark.parametrize("block", MMA_BLOCKS)
def test_mma_kernel_model_split_keeps_fp32_accuracy(P, block):
    # a model with a wide spread of magnitudes (w0 from 1e-6 to 1e3): the three bf16 rows must carry all 24 bits of
    # every entry, or the margins of the first steps are off by far more than the tolerance
    wl = wi.config3(k=4, d=2048, m=64, n_lo=40, n_hi=90)
    g = torch.Generator().manual_seed(11)
    wl.w0 = (torch.randn(2048, generator=g) * torch.logspace(-6, 3, 2048)).contiguous()
    assert_parity(P, wl, _mma(block, wl, cluster=2))


@pytest.mark.parametrize("block", MMA_BLOCKS)
def test_mma_kernel_default_shape_and_continue(P, block):
    wl_cpu = wi.small(3)
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.set_option("dense_variant", 8)
        ctx.set_option("block_samples", block)
        first = np.minimum(wl.n_steps, 301)
        ctx.run(wl.X, wl.y, wl.shard_off, first, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        ctx.continue_(wl.X, wl.y, wl.shard_off, wl.n_steps - first)
        seg = ctx.get_models().cpu().numpy()
        ctx.check()
    oW = oracle.run_dense(wl_cpu.X, wl_cpu.y, wl.shard_off, wl.n_steps, wl.d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
    for j in range(wl.k):
        assert rel_l2(seg[j], oW[j]) <= 1e-4


@pytest.mark.parametrize("block", MMA_BLOCKS)
def test_mma_kernel_limits(P, block):
    wl = wi.config2(k=2, d=64, m=16, base_steps=20)  # fp32 rows
    with pytest.raises(P.WpsgdError) as e:
        gpu_solve(P, wl, {"dense_variant": 8, "block_samples": block})
    assert e.value.status_name == "UNSUPPORTED"
    wl.X = wl.X.to(torch.bfloat16)  # 8 chunks: a cluster of 8 needs 8 non-empty slices; 16 CTAs cannot exist
    with pytest.raises(P.WpsgdError) as e:
        gpu_solve(P, wl, {"dense_variant": 8, "block_samples": block, "cluster": 16})
    assert e.value.status_name == "INVALID_ARG"


@pytest.mark.parametrize("d,cluster", [(1024, 1), (4096, 2), (4096, 4)])
@pytest.mark.parametrize("block", MMA_BLOCKS)
def test_mma_kernel_bounded_waits_report_timeout_and_context_survives(P, d, cluster, block):
    # Failure detection without a fault: the rows of block 3 are never requested (test hook), so the bounded wait
    # for them runs out; every CTA of the cluster is told, all leave in step, and the next run is clean.
    wl_cpu = wi.config2(k=3, d=d, m=32, base_steps=120)
    wl_cpu.X = wl_cpu.X.to(torch.bfloat16)
    opts = _mma(block, wl_cpu, cluster=cluster)
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        for k_, v_ in opts.items():
            ctx.set_option(k_, v_)
        ctx.set_option("spin_limit", 2000)
        ctx.set_option("test_drop_block", 3)
        ctx.run_workload(wl)
        with pytest.raises(P.WpsgdError) as e:
            ctx.check()
        assert e.value.status_name == "TIMEOUT"
        ctx.set_option("test_drop_block", -1)
        ctx.set_option("spin_limit", 1 << 20)
        ctx.run_workload(wl)
        v = ctx.combine().cpu().numpy()
        ctx.check()
    ov, _, _ = oracle.solve(wl_cpu)
    assert rel_l2(v, ov) <= 1e-4


# ---- fp32 rows, a chain spread over a cluster: variant 9, the lagged form with at most 64 chunks of a row per CTA ------------------------
@pytest.mark.parametrize("d,cluster", [(1024, 8), (1024, 4), (512, 2), (256, 1), (1000, 8), (36, 1), (2048, 8)])
@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
def test_f32_cluster_kernel_losses_and_widths(P, d, cluster, loss):
    wl = wi.config2(k=3, d=d, m=48, base_steps=210)
    wl.loss = loss
    if loss == SQUARED:
        wl.y = (wl.y * 0.3).contiguous()
    assert_parity(P, wl, {"dense_variant": 9, "cluster": cluster})


@pytest.mark.parametrize("n_steps", [(1, 7, 8), (9, 15, 16), (17, 0, 64), (333, 250, 3), (31, 32, 33)])
@pytest.mark.parametrize("cluster", [1, 4])
def test_f32_cluster_kernel_block_boundaries_and_empty_chains(P, n_steps, cluster):
    wl = wi.config2(k=3, d=256, m=64, base_steps=8)
    wl.n_steps = np.array(n_steps, dtype=np.int64)
    wl.w0 = torch.full((256,), 0.1)
    assert_parity(P, wl, {"dense_variant": 9, "cluster": cluster})


def test_f32_cluster_kernel_default_shape_and_continue(P):
    wl_cpu = wi.config2(k=5, d=1024, m=96, base_steps=700)
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.set_option("dense_variant", 9)
        first = np.minimum(wl.n_steps, 301)
        ctx.run(wl.X, wl.y, wl.shard_off, first, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        ctx.continue_(wl.X, wl.y, wl.shard_off, wl.n_steps - first)
        seg = ctx.get_models().cpu().numpy()
        ctx.check()
    oW = oracle.run_dense(wl_cpu.X, wl_cpu.y, wl.shard_off, wl.n_steps, wl.d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
    for j in range(wl.k):
        assert rel_l2(seg[j], oW[j]) <= 1e-4


def test_f32_cluster_kernel_limits(P):
    wl = wi.config2(k=2, d=2048, m=16, base_steps=20)  # 512 chunks: one CTA would hold more than 64
    with pytest.raises(P.WpsgdError) as e:
        gpu_solve(P, wl, {"dense_variant": 9, "cluster": 4})
    assert e.value.status_name == "UNSUPPORTED"
    wl.X = wl.X.to(torch.bfloat16)
    with pytest.raises(P.WpsgdError) as e:
        gpu_solve(P, wl, {"dense_variant": 9})
    assert e.value.status_name == "UNSUPPORTED"


@pytest.mark.parametrize("d,cluster", [(256, 1), (1024, 4), (1024, 8)])
def test_f32_cluster_kernel_bounded_waits_report_timeout_and_context_survives(P, d, cluster):
    # the rows of block 3 are never requested (test hook): the bounded wait for them runs out, every CTA of the
    # cluster is told, all leave in step, and the next run is clean
    wl_cpu = wi.config2(k=3, d=d, m=32, base_steps=120)
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.set_option("dense_variant", 9)
        ctx.set_option("cluster", cluster)
        ctx.set_option("spin_limit", 2000)
        ctx.set_option("test_drop_block", 3)
        ctx.run_workload(wl)
        with pytest.raises(P.WpsgdError) as e:
            ctx.check()
        assert e.value.status_name == "TIMEOUT"
        ctx.set_option("test_drop_block", -1)
        ctx.set_option("spin_limit", 1 << 20)
        ctx.run_workload(wl)
        v = ctx.combine().cpu().numpy()
        ctx.check()
    ov, _, _ = oracle.solve(wl_cpu)
    assert rel_l2(v, ov) <= 1e-4


# ---- blocked form with lagged margins (what most dense runs of up to 148 chains take) ------------------------------------
@pytest.mark.parametrize("d,bf16,pad,cluster", [
    (1, False, 0, 1), (3, True, 0, 1), (8, True, 0, 1), (36, False, 0, 1), (60, False, 0, 8),  # fewer columns than lanes
    (256, False, 0, 1), (260, False, 0, 1), (512, False, 0, 1), (516, False, 0, 1),             # 64 / 65 / 128 / 129 chunks
    (4096, False, 0, 4), (4096, False, 0, 8), (8192, True, 0, 8), (488, True, 0, 2), (2056, True, 0, 1),
    (67, False, 0, 2), (999, False, 0, 8), (1001, True, 0, 1), (1000, True, 1, 4), (640, False, 3, 2), (4099, True, 0, 8),
])
@pytest.mark.parametrize("loss,sched", [(HINGE, 0), (LOGISTIC, 1), (SQUARED, 0)])
def test_lagged_kernel_shapes(P, d, bf16, pad, cluster, loss, sched):
    # step counts with ragged last blocks, one block, none; rows that start off 16-byte boundaries (d or the row stride not
    # a multiple of 16 bytes) with garbage between the rows
    wl = wi.config2(k=4, d=d, m=48, base_steps=210)
    wl.n_steps = np.array([210, 1, 0, 67], dtype=np.int64)
    wl.loss, wl.sched = loss, sched
    if sched:
        wl.eta0, wl.lam = 0.3, 0.05
    if loss == SQUARED:
        wl.y = (wl.y * 0.3).contiguous()
    if bf16:
        wl.X = wl.X.to(torch.bfloat16)
    wl.w0 = torch.full((d,), 0.05)
    oW = oracle.run_dense(wl.X, wl.y, wl.shard_off, wl.n_steps, d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed, wl.w0)
    dev = wl.to("cuda")
    X = dev.X
    if pad:
        X = torch.full((X.shape[0], d + pad), float("nan"), dtype=X.dtype, device="cuda")
        X[:, :d] = dev.X
        X = X[:, :d]
    with P.Context(wl.k, d) as ctx:
        ctx.set_option("dense_variant", 10)
        ctx.set_option("cluster", cluster)
        ctx.run(X, dev.y, wl.shard_off, wl.n_steps, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed, dev.w0)
        W = ctx.get_models().cpu().numpy()
        ctx.check()
    for j in range(wl.k):
        assert rel_l2(W[j], oW[j]) <= TOL[loss]


@pytest.mark.parametrize("d,bf16,cluster", [
    (1024, False, 8), (1056, False, 8), (1284, False, 8), (1320, False, 8),  # 32 / 33 / 41 / 42 chunks of a CTA: 8- and 16-byte vectors, Gram warps on all schedulers
    (1024, True, 2), (1040, True, 2), (1024, True, 1), (3584, True, 2), (3600, True, 2),  # bf16: 64 / 65 / 128 / 224 / 225 chunks
    (1536, False, 2), (1544, False, 2), (3072, False, 2), (2000, False, 1),  # 192 / 193 / 384 chunks: one and two vectors per thread
    (1023, False, 4), (1025, False, 4), (1021, False, 2), (2049, True, 1),   # unaligned: 64 / 65 chunks (a block per warp, all warps per block), 128, 257
    (2047, False, 4), (3071, False, 4), (5999, False, 8), (511, False, 2), (519, False, 2),  # 64 / 65 chunks: one and two vectors per thread
])
@pytest.mark.parametrize("loss,sched", [(LOGISTIC, 0), (SQUARED, 1)])
def test_lagged_kernel_roles_at_their_limits(P, d, bf16, cluster, loss, sched):
    wl = wi.config2(k=3, d=d, m=48, base_steps=260)
    wl.n_steps = np.array([260, 129, 5], dtype=np.int64)
    wl.loss, wl.sched = loss, sched
    if loss == SQUARED:
        wl.y = (wl.y * 0.3).contiguous()
    if bf16:
        wl.X = wl.X.to(torch.bfloat16)
    if (d * (2 if bf16 else 4) + 15) // 16 > (256 if d % 2 else 512) * cluster:
        with pytest.raises(P.WpsgdError):  # more chunks of a row than the CTAs take
            gpu_solve(P, wl, {"dense_variant": 10, "cluster": cluster})
        return
    assert_parity(P, wl, {"dense_variant": 10, "cluster": cluster})


@pytest.mark.parametrize("d,bf16,cluster,stages", [
    (3592, False, 2, 0), (4096, False, 2, 0), (8192, True, 2, 0),  # 449 / 512 chunks of a CTA, eight model warps: one team, a ring of 3
    (2045, True, 2, 3), (2045, True, 2, 6), (1567, True, 2, 0),    # unaligned, 128 / 98 chunks: one team on 3 stages, three on 6 and 12
    (1023, True, 2, 0), (799, True, 2, 0), (3711, True, 8, 0),     # a block per realigning warp, 64 / 50 / 58 chunks: rings of 12, 12 and 8
    (4093, True, 2, 0), (2045, False, 2, 0),                       # 256 chunks, a ring of 3
])
@pytest.mark.parametrize("loss,sched", [(LOGISTIC, 0), (SQUARED, 1)])
def test_lagged_kernel_teams_of_three_gram_warps(P, d, bf16, cluster, stages, loss, sched):
    wl = wi.config2(k=3, d=d, m=48, base_steps=330)
    wl.n_steps = np.array([330, 129, 5], dtype=np.int64)
    wl.loss, wl.sched = loss, sched
    if loss == SQUARED:
        wl.y = (wl.y * 0.3).contiguous()
    if bf16:
        wl.X = wl.X.to(torch.bfloat16)
    assert_parity(P, wl, {"dense_variant": 10, "cluster": cluster, "stages": stages})


@pytest.mark.parametrize("k", [3, 240])  # tables as an argument of the stream kernel, and copied
def test_runs_in_a_row_do_not_read_each_others_streams(P, k):
    # the stream of a run is formed while kernels before it are still at work; a run that is refused after its stream was
    # launched must not disturb the next one
    wl = wi.config2(k=k, d=40, m=32, base_steps=90).to("cuda")
    want = []
    for seed in (1, 2):
        with P.Context(wl.k, wl.d) as ctx:
            wl.seed = seed
            ctx.run_workload(wl)
            want.append(ctx.combine().cpu().numpy())
    with P.Context(wl.k, wl.d) as ctx:
        for rep in range(6):
            wl.seed = 1 + rep % 2
            if rep >= 2:
                ctx.set_option("dense_variant", 8)  # fp32 rows: refused
                with pytest.raises(P.WpsgdError):
                    ctx.run_workload(wl)
                ctx.set_option("dense_variant", 0)
            ctx.run_workload(wl)
            v = ctx.combine()
            np.testing.assert_array_equal(v.cpu().numpy(), want[rep % 2])


@pytest.mark.parametrize("variant,bf16,stride", [(9, False, 2 ** 31), (10, False, 2 ** 31 + 4), (10, True, 2 ** 32 + 16), (0, False, 2 ** 31 + 16)])
def test_lagged_kernel_takes_row_strides_of_2_gib_and_more(P, variant, bf16, stride):
    # three rows, 2 or 4 GiB apart (the third one beyond what 32 bits of a byte offset hold); rows off 16-byte boundaries too
    wl = wi.config2(k=1, d=40, m=3, base_steps=40)
    if bf16:
        wl.X = wl.X.to(torch.bfloat16)
    oW = oracle.run_dense(wl.X, wl.y, wl.shard_off, wl.n_steps, wl.d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
    dev = wl.to("cuda")
    ld = stride // wl.X.element_size()
    X = torch.empty(2 * ld + 64, dtype=wl.X.dtype, device="cuda").as_strided((3, 40), (ld, 1))
    X.copy_(dev.X)
    with P.Context(wl.k, wl.d) as ctx:
        ctx.set_option("dense_variant", variant)
        ctx.run(X, dev.y, wl.shard_off, wl.n_steps, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        W = ctx.get_models().cpu().numpy()
        ctx.check()
    assert rel_l2(W[0], oW[0]) <= TOL[wl.loss]


def test_a_failed_allocation_does_not_fail_the_next_call(P):
    wl = wi.config2(k=2, d=40, m=16, base_steps=40).to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        with pytest.raises(P.WpsgdError) as e:  # a sample stream of 1.6 TB
            ctx.run(wl.X, wl.y, wl.shard_off, np.array([200 * 10 ** 9] * 2, dtype=np.int64), wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        assert e.value.status_name == "ALLOC"
        ctx.run_workload(wl)
        ctx.check()


def test_contexts_of_two_threads_launch_one_kernel_with_different_shared_memory(P):
    # the limit on a kernel's shared memory belongs to the process: the launch of a large ring must not meet the limit of a small one
    import ctypes
    import threading

    failed = []

    def work(d, stages):
        X, y = torch.randn(16, d, device="cuda"), torch.ones(16, device="cuda")
        n, off = np.array([8], dtype=np.int64), np.array([0, 16], dtype=np.int64)
        with torch.cuda.stream(torch.cuda.Stream()), P.Context(1, d) as ctx:
            ctx.set_option("dense_variant", 10)
            ctx.set_option("cluster", 1)
            ctx.set_option("stages", stages)
            args = (ctx._h, ctypes.c_void_p(X.data_ptr()), P.X_F32, d, ctypes.c_void_p(y.data_ptr()), off.ctypes.data, n.ctypes.data, 0.01,
                    P.LR_CONST, 1e-4, P.LOSS_SQUARED, 1, None)
            for i in range(3000):  # the bare entry point: little between two calls but the launch
                if ctx._lib.wpsgd_run(*args):
                    failed.append((d, i, ctx._lib.wpsgd_last_error(ctx._h).decode()))
                if i % 64 == 0:
                    torch.cuda.current_stream().synchronize()
            ctx.check()

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=a) for a in ((160, 3), (960, 6))]  # one form of the kernel, about 30 and 200 KB
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, (len(failed), failed[:3])


@pytest.mark.parametrize("k,chunks,cluster", [(74, 392, 2), (4, 416, 1), (4, 372, 4)])
def test_slices_that_fill_shared_memory_keep_a_ring_of_four_stages(P, k, chunks, cluster):
    # with a ring of three the lagged kernel is not offered (unless its cluster size is asked for): 74 chains took a direct kernel
    # and 1470 us instead of 213. What is asked for is what runs by itself.
    wl = wi.config3(k=k, d=8 * chunks * cluster, m=16, n_lo=800 if k == 74 else 40, n_hi=800 if k == 74 else 40)
    if cluster != 2:  # few chains would take more CTAs
        assert_parity(P, wl, {"dense_variant": 10, "cluster": cluster, "stages": 4})
        return
    np.testing.assert_array_equal(gpu_solve(P, wl)[0], gpu_solve(P, wl, {"dense_variant": 10, "cluster": cluster})[0])


@pytest.mark.parametrize("k,d,steps", [(4, 64, 128), (148, 128, 128), (37, 256, 256), (4, 1000, 128)])
def test_short_runs_of_few_bf16_chains_take_the_lagged_kernel(P, k, d, steps):
    # 14 to 25 us there, 25 to 70 % more in the kernels that share the shape (and other bits: their sums are in another order)
    wl = wi.config3(k=k, d=d, m=16, n_lo=steps, n_hi=steps)
    np.testing.assert_array_equal(gpu_solve(P, wl)[0], gpu_solve(P, wl, {"dense_variant": 10})[0])


@pytest.mark.parametrize("stages", [0, 3, 4, 5])
@pytest.mark.parametrize("n_steps", [(1, 7, 8), (9, 15, 16), (17, 0, 64), (333, 250, 3)])
def test_lagged_kernel_block_boundaries_and_ring_depths(P, n_steps, stages):
    wl = wi.config2(k=3, d=1024, m=64, base_steps=8)
    wl.n_steps = np.array(n_steps, dtype=np.int64)
    wl.w0 = torch.full((1024,), 0.1)
    assert_parity(P, wl, {"dense_variant": 10, "cluster": 2, "stages": stages})


@pytest.mark.parametrize("d,cluster", [(64, 1), (1024, 4), (999, 8)])
def test_lagged_kernel_bounded_waits_report_timeout_and_context_survives(P, d, cluster):
    wl_cpu = wi.config2(k=3, d=d, m=32, base_steps=120)
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        for name, value in (("dense_variant", 10), ("cluster", cluster), ("spin_limit", 2000), ("test_drop_block", 3)):
            ctx.set_option(name, value)
        ctx.run_workload(wl)
        with pytest.raises(P.WpsgdError) as e:
            ctx.check()
        assert e.value.status_name == "TIMEOUT"
        ctx.set_option("test_drop_block", -1)
        ctx.set_option("spin_limit", 1 << 20)
        ctx.run_workload(wl)
        v = ctx.combine().cpu().numpy()
        ctx.check()
    ov, _, _ = oracle.solve(wl_cpu)
    assert rel_l2(v, ov) <= 1e-4


# ---- logistic loss: blocks whose steps move the margins far take the direct evaluation ---------------------------------
@pytest.mark.parametrize("variant,d", [(4, 1024), (5, 128), (8, 1024), (9, 1024), (10, 200)])
def test_logistic_large_steps_between_correlated_rows(P, variant, d):
    # rows that are nearly parallel (large Gram entries) and a large step size: inside a block of 8 samples the
    # margins move by much more than the range of the cubic expansion of the logistic factor
    wl = wi.config2(k=3, d=d, m=64, base_steps=160)
    g = torch.Generator().manual_seed(5)
    base = torch.randn(d, generator=g) / np.sqrt(d)
    wl.X = (2.0 * base[None, :] + 0.3 * wl.X).contiguous()
    wl.eta0 = 0.4
    if variant == 8:
        wl.X = wl.X.to(torch.bfloat16)
    assert_parity(P, wl, {"dense_variant": variant})


@pytest.mark.parametrize("k,variant", [(4, 9), (40, 4)])
def test_default_kernels_for_large_aligned_fp32_rows(P, k, variant):
    # few chains: each spread over a cluster of idle SMs (lagged form); many chains: one CTA each
    wl = wi.config2(k=k, d=1024, m=64, base_steps=100).to("cuda")
    with P.Context(wl.k, wl.d) as a, P.Context(wl.k, wl.d) as b:
        a.run_workload(wl)
        b.set_option("dense_variant", variant)
        b.run_workload(wl)
        np.testing.assert_array_equal(a.get_models().cpu().numpy(), b.get_models().cpu().numpy())
        a.check()
        b.check()


def test_tensor_core_cluster_kernel_is_the_default_for_wide_bf16_rows(P):
    wl = wi.config3(k=4, d=2048, m=64, n_lo=60, n_hi=120).to("cuda")
    with P.Context(wl.k, wl.d) as a, P.Context(wl.k, wl.d) as b:
        a.run_workload(wl)
        b.set_option("dense_variant", 8)
        b.run_workload(wl)
        np.testing.assert_array_equal(a.get_models().cpu().numpy(), b.get_models().cpu().numpy())
        a.check()
        b.check()


def _models(P, wl, **opts):
    with P.Context(wl.k, wl.d) as ctx:
        for name, value in opts.items():
            ctx.set_option(name, value)
        ctx.run_workload(wl)
        W = ctx.get_models().cpu().numpy()
        ctx.check()
    return W


def test_dense_variant_8_forces_the_tensor_core_kernel(P):
    # few chains of 1000 steps: variant 10 is the default there, and an explicit 8 is not
    wl = wi.config3(k=3, d=1024, m=64, n_lo=1000, n_hi=1000).to("cuda")
    W8 = _models(P, wl, dense_variant=8)
    np.testing.assert_array_equal(W8, _models(P, wl, dense_variant=8, block_samples=16))
    W10 = _models(P, wl, dense_variant=10)
    assert not np.array_equal(W8, W10)
    np.testing.assert_array_equal(_models(P, wl), W10)


def test_default_kernels_far_from_the_crossover(P):
    # every form sums in another order, so equal bits name the kernel
    wide = wi.config3(k=128, d=4096, m=16, n_lo=60, n_hi=120).to("cuda")
    W = _models(P, wide)
    np.testing.assert_array_equal(W, _models(P, wide, dense_variant=8, block_samples=16))
    assert not np.array_equal(W, _models(P, wide, dense_variant=10))
    few = wi.config2(k=4, d=1024, m=64, base_steps=400).to("cuda")
    W = _models(P, few)
    np.testing.assert_array_equal(W, _models(P, few, dense_variant=10))
    assert not np.array_equal(W, _models(P, few, dense_variant=4))


# ---- degenerate cases -----------------------------------------------------------------------------------
def test_nodes_without_work_keep_w0(P):
    wl = wi.config1(k=4, d=64, m=64, n_steps=(120, 0, 30, 0))
    wl.w0 = torch.full((64,), 4.0)  # the paper's experiments start from the constant vector 4
    v, W, wts, _ = gpu_solve(P, wl)
    assert np.all(W[1] == 4.0) and np.all(W[3] == 4.0)
    assert_parity(P, wl)


@pytest.mark.parametrize("sampling", [0, 1])
@pytest.mark.parametrize("d,bf16,loss,opts", [
    (999, False, SQUARED, {}), (999, False, LOGISTIC, {}), (999, False, HINGE, {}), (1000, True, HINGE, {}), (64, False, HINGE, {}),
    (8192, False, LOGISTIC, {}), (1024, False, SQUARED, {"dense_variant": 4}), (128, False, SQUARED, {"dense_variant": 5}),
    (4096, True, SQUARED, {"dense_variant": 8, "block_samples": 16}), (4096, True, LOGISTIC, {"dense_variant": 8, "block_samples": 8}),
])
def test_rows_that_no_step_visits_do_not_reach_the_model(P, d, bf16, loss, opts, sampling):
    # 21 steps end inside a block of 8 or 16: what fills the block up must not bring in other rows (here NaN) or labels
    wl = wi.config2(k=2, d=d, m=512, base_steps=21)
    wl.n_steps = np.array([21, 1], dtype=np.int64)
    wl.loss = loss
    if loss == SQUARED:
        wl.y = (wl.y * 0.3).contiguous()
    if bf16:
        wl.X = wl.X.to(torch.bfloat16)
    opts = dict(opts, sampling=sampling)
    _, clean, _, _ = gpu_solve(P, wl, opts)
    unseen = torch.ones(len(wl.y), dtype=torch.bool)
    for j in range(2):
        rows = P.sample_indices_host(wl.seed, j, 512, 0, int(wl.n_steps[j]), sampling).astype(np.int64) + int(wl.shard_off[j])
        unseen[torch.from_numpy(rows)] = False
    wl.X, wl.y = wl.X.clone(), wl.y.clone()
    wl.X[unseen] = float("nan")
    wl.y[unseen] = float("nan")
    _, W, _, _ = gpu_solve(P, wl, opts)
    np.testing.assert_array_equal(W, clean)


def test_no_work_at_all_returns_w0(P):
    wl = wi.config1(k=3, d=64, m=8, n_steps=(0, 0, 0))
    wl.w0 = torch.arange(64, dtype=torch.float32)
    v, W, wts, _ = gpu_solve(P, wl)
    np.testing.assert_array_equal(wts, np.full(3, 1 / 3))
    np.testing.assert_allclose(v, np.arange(64), rtol=1e-6)
    wl.w0 = None
    v, W, _, _ = gpu_solve(P, wl)
    assert np.all(v == 0) and np.all(W == 0)


def test_single_node_is_sequential_sgd(P):
    wl = wi.config1(k=1, d=64, m=256, n_steps=(500,))
    v, W, wts, flag = gpu_solve(P, wl)
    assert wts[0] == 1.0 and flag is False  # Eq. 7 with k = 1: 2 > 2 is false
    np.testing.assert_array_equal(v, W[0])
    assert_parity(P, wl)


def test_single_row_shards_and_unequal_shards(P):
    g = torch.Generator().manual_seed(5)
    d = 32
    off = np.array([0, 1, 4, 4, 40], dtype=np.int64)  # shard sizes 1, 3, 0, 36
    X = torch.randn(40, d, generator=g) / 4
    y = torch.sign(torch.randn(40, generator=g))
    n = np.array([25, 60, 0, 100], dtype=np.int64)
    wl = wi.Workload("ragged", 4, d, off, n, 0.05, 0, 0.01, LOGISTIC, 9, y, X=X)
    assert_parity(P, wl)
    for variant in (1, 2, 3):
        assert_parity(P, wl, {"dense_variant": variant})


def test_equal_work_reduces_to_plain_average(P):
    wl = wi.config2(k=6, d=128, m=64, base_steps=90)
    wl.n_steps[:] = 90
    v, W, wts, _ = gpu_solve(P, wl)
    np.testing.assert_array_equal(wts, np.full(6, 1 / 6))
    np.testing.assert_allclose(v, W.astype(np.float64).mean(0), rtol=1e-6, atol=1e-9)


def test_relabelling_a_node_changes_only_its_stream(P):
    # the same shard at node position j must see the oracle's stream for node j
    wl = wi.config1(k=3, d=64, m=64, n_steps=(50, 50, 50))
    _, W, _, _ = gpu_solve(P, wl)
    assert not np.array_equal(W[0], W[1])
    assert_parity(P, wl)


# ---- combination --------------------------------------------------------------------------------------
@pytest.mark.parametrize("r", [0.0, 1.0, 0.99999, 0.9])
def test_combine_rates(P, r):
    wl = wi.config1(k=4, d=64, m=64, n_steps=(400, 300, 100, 7))
    v, W, wts, flag = gpu_solve(P, wl, r=r)
    owts, oflag, _ = oracle.weights(wl.n_steps, wl.eta0, wl.sched, wl.lam, r)
    np.testing.assert_allclose(wts, owts, rtol=1e-12)
    assert flag == oflag
    want = oracle.combine(W.astype(np.float64), owts)  # the GPU's own models, so this isolates the reduction
    np.testing.assert_allclose(v, want, rtol=2e-7, atol=1e-12)


def test_combine_many_nodes_ragged_d(P):
    k, d = 37, 1001
    g = torch.Generator().manual_seed(1)
    X = torch.randn(k * 4, d, generator=g)
    y = torch.sign(torch.randn(k * 4, generator=g))
    n = (np.arange(k) % 5).astype(np.int64)
    wl = wi.Workload("wide", k, d, np.arange(k + 1, dtype=np.int64) * 4, n, 0.01, 0, 0.1, HINGE, 2, y, X=X)
    assert_parity(P, wl)


# ---- segmented runs and periodic averaging ----------------------------------------------------------------
def test_continue_blocked_kernel(P):
    # the blocked kernel groups samples by eight from wherever a segment starts, so a cut run agrees with the
    # uncut one up to rounding order (not bit for bit)
    wl_cpu = wi.config2(k=3, d=256, m=128, base_steps=203)
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.set_option("dense_variant", 4)
        first = np.minimum(wl.n_steps, 37)
        ctx.run(wl.X, wl.y, wl.shard_off, first, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        ctx.continue_(wl.X, wl.y, wl.shard_off, wl.n_steps - first)
        seg = ctx.get_models().cpu().numpy()
        ctx.check()
    oW = oracle.run_dense(wl_cpu.X, wl_cpu.y, wl.shard_off, wl.n_steps, wl.d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
    for j in range(wl.k):
        assert rel_l2(seg[j], oW[j]) <= 1e-4


@pytest.mark.parametrize("variant", [1, 2, 3])
def test_continue_equals_one_run(P, variant):
    wl = wi.config1(k=3, d=64, m=128, n_steps=(203, 101, 50)).to("cuda")
    wl.sched = 1  # the step number matters for eta_n, so a wrong restart shows
    with P.Context(wl.k, wl.d) as ctx:
        ctx.set_option("dense_variant", variant)
        ctx.run_workload(wl)
        full = ctx.get_models().cpu().numpy()
        cuts = [np.array([50, 50, 50]), np.array([1, 1, 0]), np.array([152, 50, 0])]
        ctx.run(wl.X, wl.y, wl.shard_off, cuts[0], wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        for c in cuts[1:]:
            ctx.continue_(wl.X, wl.y, wl.shard_off, c)
        seg = ctx.get_models().cpu().numpy()
        wts, _ = ctx.get_weights()
        ctx.check()
    np.testing.assert_array_equal(seg, full)  # same arithmetic in the same order
    owts, _, _ = oracle.weights(wl.n_steps, wl.eta0, wl.sched, wl.lam)
    np.testing.assert_allclose(wts, owts, rtol=1e-12)


def test_periodic_weighted_averaging(P):
    # average every `span` fastest-node steps, then continue from the average on every node
    wl = wi.config2(k=4, d=128, m=64, base_steps=120)
    span_steps = [np.array([40, 20, 10, 40]), np.array([40, 20, 10, 40]), np.array([40, 20, 10, 40])]
    dev = wl.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.run(dev.X, dev.y, wl.shard_off, span_steps[0], wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        for seg in span_steps[1:]:
            ctx.set_models(ctx.combine())
            ctx.continue_(dev.X, dev.y, wl.shard_off, seg)
        v = ctx.combine().cpu().numpy()
        ctx.check()
    # oracle: same schedule; weights of each round come from that round's step counts
    W = oracle.run_dense(wl.X, wl.y, wl.shard_off, span_steps[0], wl.d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
    done = span_steps[0].copy()
    for seg in span_steps[1:]:
        wts, _, _ = oracle.weights(done, wl.eta0, wl.sched, wl.lam)
        vv = oracle.combine(W, wts)
        # steps continue from each node's own count: run node by node with its own step_begin
        Wn = np.zeros_like(W)
        for j in range(wl.k):
            only = np.zeros(wl.k, dtype=np.int64)
            only[j] = seg[j]
            Wn[j] = oracle.run_dense(wl.X, wl.y, wl.shard_off, only, wl.d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed,
                                     step_begin=int(done[j]), W_resume=np.tile(vv.astype(np.float32).astype(np.float64), (wl.k, 1)))[j]
        W = Wn
        done = done + seg
    wts, _, _ = oracle.weights(done, wl.eta0, wl.sched, wl.lam)
    assert rel_l2(v, oracle.combine(W, wts)) <= 1e-4


# ---- evaluation measures ---------------------------------------------------------------------------------
@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
@pytest.mark.parametrize("bf16", [False, True])
def test_objective_and_error_rate(P, loss, bf16):
    wl = wi.config1(k=2, d=64, m=333, n_steps=(10, 10))
    X = wl.X.to(torch.bfloat16) if bf16 else wl.X
    w = (torch.randn(64, generator=torch.Generator().manual_seed(4)) / 8)
    with P.Context(2, 64) as ctx:
        out = ctx.objective(X.cuda(), wl.y.cuda(), w.cuda(), 0.01, loss).cpu().numpy()
        ctx.check()
    obj, err = oracle.objective_dense(X, wl.y, w.numpy().astype(np.float64), 0.01, loss)
    assert out[0] == pytest.approx(obj, rel=1e-5)
    assert abs(out[1] - err) <= 2.0 / 666  # a margin within fp32 rounding of 0 may flip


@pytest.mark.parametrize("d", [1, 31, 33, 64, 65, 96, 97, 128, 129, 160, 161, 256, 257, 264, 520])
@pytest.mark.parametrize("bf16,shift", [(False, 0), (True, 0), (False, 1)])
def test_objective_row_widths(P, d, bf16, shift):
    # around the ends of the loads in flight: 32 and 128 chunks of 16 bytes, 64 and 128 single elements; rows that start off 16
    # bytes (shift); row counts that leave warps with one to four rows in flight (37) and with several turns of them (40000)
    for rows in (37, 40000 if d <= 64 else 9600):
        g = torch.Generator().manual_seed(d)
        X = torch.randn(rows * d + shift, generator=g)
        X = (X.to(torch.bfloat16) if bf16 else X)
        w = torch.randn(d, generator=g) / np.sqrt(d)
        y = torch.sign(torch.randn(rows, generator=g))
        with P.Context(1, d) as ctx:
            out = ctx.objective(X.cuda()[shift:].view(rows, d), y.cuda(), w.cuda(), 0.01, LOGISTIC).cpu().numpy()
            ctx.check()
        Xr = X[shift:].view(rows, d).contiguous()
        obj, err = oracle.objective_dense(Xr, y, w.numpy().astype(np.float64), 0.01, LOGISTIC)
        # the rounding of a margin (some units of 2^-24 of sum |w x|) is of either sign and averages out over the rows
        assert out[0] == pytest.approx(obj, rel=1e-6)
        assert abs(out[1] - err) <= 2.0 / rows


@pytest.mark.parametrize("rows", [1, 300, 4736, 4737])
def test_objective_csr_rows_of_all_lengths(P, rows):
    # 4736 rows are the most that get a warp each; above, four rows share a warp unless one is longer than 512
    g = torch.Generator().manual_seed(rows)
    d = 3000
    kinds = [0, 1, 7, 8, 33, 127, 128, 129] + [2] * 20
    lengths = [kinds[i % len(kinds)] for i in range(rows)]
    for i, n in ((0, 513), (5, 512), (9, 2900), (rows - 1, 1025)):
        if i < rows:
            lengths[i] = n
    rp = torch.zeros(rows + 1, dtype=torch.int64)
    rp[1:] = torch.cumsum(torch.tensor(lengths), 0)
    ci = torch.cat([torch.sort(torch.randint(0, d, (n,), generator=g))[0] for n in lengths]).to(torch.int32)
    va = torch.randn(len(ci), generator=g) / 8
    y = torch.sign(torch.randn(rows, generator=g))
    w = torch.randn(d, generator=g)
    with P.Context(1, d) as ctx:
        out = ctx.objective_csr(rp.cuda(), ci.cuda(), va.cuda(), y.cuda(), w.cuda(), 0.01, SQUARED).cpu().numpy()
        ctx.check()
    obj, err = oracle.objective_csr(rp, ci, va, y, w.numpy().astype(np.float64), 0.01, SQUARED)
    assert out[0] == pytest.approx(obj, rel=1e-6)
    assert abs(out[1] - err) <= 2.0 / rows


# ---- host-buffer entry point --------------------------------------------------------------------------------
def test_solve_host_equals_device_path(P):
    wl = wi.config2(k=5, d=256, m=128, base_steps=200)
    wl.w0 = torch.full((256,), 0.5)
    v_dev, _, _, _ = gpu_solve(P, wl)
    with P.Context(wl.k, wl.d) as ctx:
        out = ctx.solve_host(wl.X.pin_memory(), wl.y.pin_memory(), wl.shard_off, wl.n_steps, wl.eta0, wl.sched, wl.lam,
                             wl.loss, wl.seed, w0=wl.w0)
        again = ctx.solve_host(wl.X, wl.y, wl.shard_off, wl.n_steps, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed,
                               w0=wl.w0)  # pageable source, buffers reused
        ctx.check()
    np.testing.assert_array_equal(out.numpy(), v_dev)
    np.testing.assert_array_equal(again.numpy(), v_dev)


@pytest.mark.parametrize("d,bf16,k", [(1024, False, 5), (1024, False, 2), (2048, True, 7), (480, False, 3)])
@pytest.mark.parametrize("pipeline", [0, 1])
def test_solve_host_pipelined_equals_device_path(P, d, bf16, k, pipeline):
    # rows wide enough for the pipelined form: shards copied in groups (longest chains first), chains of a group
    # launched when its rows have arrived; the per-node arithmetic is the same, so the result is bit for bit that of
    # the device path
    wl = wi.config2(k=k, d=d, m=96, base_steps=230)
    wl.n_steps[k - 1] = 0
    if bf16:
        wl.X = wl.X.to(torch.bfloat16)
    wl.w0 = torch.full((d,), 0.25)
    v_dev, _, _, _ = gpu_solve(P, wl)
    with P.Context(wl.k, wl.d) as ctx:
        ctx.set_option("host_pipeline", pipeline)
        for _ in range(2):
            out = ctx.solve_host(wl.X.pin_memory(), wl.y.pin_memory(), wl.shard_off, wl.n_steps, wl.eta0, wl.sched, wl.lam,
                                 wl.loss, wl.seed, w0=wl.w0)
            np.testing.assert_array_equal(out.numpy(), v_dev)
        ctx.check()


def test_solve_host_pipelined_groups_take_the_kernel_of_their_own_size(P):
    # 64 chains in four launches of 16: each launch has the GPU to itself and has to run what a context of these 16 nodes
    # runs (a cluster of CTAs per chain), not what 64 chains at once would take (one CTA per chain)
    wl = wi.config2(k=64, d=1024, m=48, base_steps=8)
    wl.n_steps = 420 - np.arange(64, dtype=np.int64)
    dev = wl.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.solve_host(wl.X.pin_memory(), wl.y.pin_memory(), wl.shard_off, wl.n_steps, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        W = ctx.get_models().cpu().numpy()
        ctx.check()
    for g in range(0, 64, 16):
        lo, hi = int(wl.shard_off[g]), int(wl.shard_off[g + 16])
        with P.Context(16, wl.d) as ctx:
            ctx.set_node_ids(np.arange(g, g + 16))
            ctx.run(dev.X[lo:hi], dev.y[lo:hi], wl.shard_off[g:g + 17] - lo, wl.n_steps[g:g + 16], wl.eta0, wl.sched, wl.lam, wl.loss,
                    wl.seed)
            np.testing.assert_array_equal(W[g:g + 16], ctx.get_models().cpu().numpy())
            ctx.check()


def test_solve_host_csr_equals_device_path(P):
    wl = wi.config4(k=5, d=4096, m=200, base_steps=500, mean_nnz=25.0)
    wl.w0 = torch.full((4096,), 0.02)
    v_dev, _, _, _ = gpu_solve(P, wl)
    with P.Context(wl.k, wl.d) as ctx:
        for _ in range(2):
            out = ctx.solve_host_csr(wl.row_ptr.pin_memory(), wl.col_idx.pin_memory(), wl.val.pin_memory(), wl.y.pin_memory(),
                                     wl.shard_off, wl.n_steps, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed, w0=wl.w0)
            np.testing.assert_array_equal(out.numpy(), v_dev)
        ctx.check()
    ov, _, _ = oracle.solve(wl)
    assert rel_l2(out.numpy(), ov) <= TOL[wl.loss]


# ---- sparse path --------------------------------------------------------------------------------------------
# sparse_variant 1: one step per round trip to the model in global memory; 2 (the default): blocks of steps run in a
# shared-memory cache of the model entries they touch
@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
@pytest.mark.parametrize("variant,prefetch", [(1, 2), (1, 4), (1, 8), (2, 0)])
def test_csr_losses_and_kernels(P, loss, variant, prefetch):
    wl = wi.config4(k=5, d=4096, m=300, base_steps=700, mean_nnz=30.0)
    wl.loss = loss
    if loss == SQUARED:
        wl.eta0 = 0.05
    wl.w0 = torch.full((4096,), 0.01)
    assert_parity(P, wl, {"sparse_variant": variant, "prefetch": prefetch})


@pytest.mark.parametrize("variant", [1, 2])
def test_csr_long_rows_and_strong_regulariser(P, variant):
    # rows with up to 128 nonzeros (beyond the 64 kept in registers); eta*lambda large enough that the
    # scale factor is folded back into the model several times
    wl = wi.config4(k=3, d=512, m=64, base_steps=400, mean_nnz=90.0, max_nnz=128)
    wl.sched, wl.eta0, wl.lam = 0, 0.5, 0.5  # (1 - 0.25)^400 ~ 1e-50
    wl.w0 = torch.full((512,), 1.0)
    assert_parity(P, wl, {"sparse_variant": variant})


@pytest.mark.parametrize("n_steps", [(1, 63, 64), (65, 127, 128), (129, 0, 200), (333, 250, 3)])
@pytest.mark.parametrize("mean_nnz", [8.0, 100.0])
def test_csr_block_kernel_block_boundaries(P, n_steps, mean_nnz):
    # short rows: a block ends after 64 steps; long rows: it ends when its 4096 table entries are used up
    wl = wi.config4(k=3, d=2048, m=96, base_steps=10, mean_nnz=mean_nnz, max_nnz=128)
    wl.n_steps = np.array(n_steps, dtype=np.int64)
    wl.w0 = torch.full((2048,), 0.02)
    assert_parity(P, wl, {"sparse_variant": 2})


def _rows_with_given_lengths(lengths, d, seed):
    """Hand-built CSR rows of the given lengths: distinct sorted random columns, values 1/sqrt(nnz), labels +-1."""
    g = torch.Generator().manual_seed(seed)
    cols, vals = [], []
    for n in lengths:
        c, _ = torch.sort(torch.randperm(d, generator=g)[:n])
        cols.append(c.to(torch.int32))
        vals.append(torch.full((n,), 1.0 / np.sqrt(max(n, 1))))
    rp = torch.zeros(len(lengths) + 1, dtype=torch.int64)
    rp[1:] = torch.cumsum(torch.tensor(lengths), 0)
    y = torch.where(torch.rand(len(lengths), generator=g) < 0.5, 1.0, -1.0)
    return rp, torch.cat(cols), torch.cat(vals), y


@pytest.mark.parametrize("loss", [HINGE, SQUARED])
def test_csr_rows_longer_than_the_block_tables(P, loss):
    # rows of 5000 and 6000 nonzeros do not fit the 4096 table entries of a block: such a step is run on global
    # memory, between ordinary blocks of short rows
    d = 8192
    lengths = [5000, 12, 30, 6000, 7, 4096, 4097, 64, 1, 0, 33, 65]
    rp, ci, va, y = _rows_with_given_lengths(lengths, d, 11)
    wl = wi.Workload("long", 2, d, np.array([0, 6, 12]), np.array([150, 90]), 0.2, 1, 0.01, loss, 5, y, row_ptr=rp,
                     col_idx=ci, val=va, w0=torch.full((d,), 0.01))
    assert_parity(P, wl, {"sparse_variant": 2})


@pytest.mark.parametrize("variant", [1, 2])
def test_continue_csr_equals_one_run(P, variant):
    wl_cpu = wi.config4(k=3, d=4096, m=128, base_steps=10, mean_nnz=30.0)
    wl_cpu.n_steps = np.array([203, 101, 50], dtype=np.int64)
    wl_cpu.lam = 0.01
    wl = wl_cpu.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.set_option("sparse_variant", variant)
        ctx.run_workload(wl)
        full = ctx.get_models().cpu().numpy()
        cuts = [np.array([50, 50, 50]), np.array([1, 1, 0]), np.array([152, 50, 0])]
        ctx.run_csr(wl.row_ptr, wl.col_idx, wl.val, wl.y, wl.shard_off, cuts[0], wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
        for c in cuts[1:]:
            ctx.continue_csr(wl.row_ptr, wl.col_idx, wl.val, wl.y, wl.shard_off, c)
        seg = ctx.get_models().cpu().numpy()
        wts, _ = ctx.get_weights()
        ctx.check()
    if variant == 1:
        np.testing.assert_array_equal(seg, full)  # same arithmetic in the same order
    else:
        # the fp64 scale is a product over the steps of a block, so cutting the chain changes its last bits only
        for j in range(wl.k):
            assert rel_l2(seg[j], full[j]) <= 1e-6
    owts, _, _ = oracle.weights(wl_cpu.n_steps, wl_cpu.eta0, wl_cpu.sched, wl_cpu.lam)
    np.testing.assert_allclose(wts, owts, rtol=1e-12)
    oW = oracle.run_csr(wl_cpu.row_ptr, wl_cpu.col_idx, wl_cpu.val, wl_cpu.y, wl_cpu.shard_off, wl_cpu.n_steps, wl_cpu.d,
                        wl_cpu.eta0, wl_cpu.sched, wl_cpu.lam, wl_cpu.loss, wl_cpu.seed)
    for j in range(wl.k):
        assert rel_l2(seg[j], oW[j]) <= TOL[wl_cpu.loss]


def test_periodic_weighted_averaging_on_csr_rows(P):
    # average every span of fastest-node steps, broadcast, continue: the paper's bucket-style WP-SGD on sparse rows.
    # The checker runs the same schedule on the densified rows (its dense loop can start from a given model and step).
    wl = wi.config4(k=4, d=256, m=64, base_steps=10, mean_nnz=12.0, max_nnz=32)
    wl.loss, wl.sched, wl.eta0, wl.lam = LOGISTIC, 0, 0.1, 0.01
    span_steps = [np.array([40, 20, 10, 40]), np.array([40, 20, 10, 40]), np.array([40, 20, 10, 40])]
    dev = wl.to("cuda")
    with P.Context(wl.k, wl.d) as ctx:
        ctx.run_csr(dev.row_ptr, dev.col_idx, dev.val, dev.y, wl.shard_off, span_steps[0], wl.eta0, wl.sched, wl.lam,
                    wl.loss, wl.seed)
        for seg in span_steps[1:]:
            ctx.set_models(ctx.combine())
            ctx.continue_csr(dev.row_ptr, dev.col_idx, dev.val, dev.y, wl.shard_off, seg)
        v = ctx.combine().cpu().numpy()
        ctx.check()
    dn = wi.densify(wl)
    W = oracle.run_dense(dn.X, dn.y, wl.shard_off, span_steps[0], wl.d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed)
    done = span_steps[0].copy()
    for seg in span_steps[1:]:
        wts, _, _ = oracle.weights(done, wl.eta0, wl.sched, wl.lam)
        vv = oracle.combine(W, wts)
        Wn = np.zeros_like(W)
        for j in range(wl.k):
            only = np.zeros(wl.k, dtype=np.int64)
            only[j] = seg[j]
            Wn[j] = oracle.run_dense(dn.X, dn.y, wl.shard_off, only, wl.d, wl.eta0, wl.sched, wl.lam, wl.loss, wl.seed,
                                     step_begin=int(done[j]),
                                     W_resume=np.tile(vv.astype(np.float32).astype(np.float64), (wl.k, 1)))[j]
        W = Wn
        done = done + seg
    wts, _, _ = oracle.weights(done, wl.eta0, wl.sched, wl.lam)
    assert rel_l2(v, oracle.combine(W, wts)) <= 1e-4


def test_validate_csr_accepts_good_input_and_names_the_bad_row(P):
    # the malformed arrays below are only ever read by the validator (which reads nothing outside [0, nnz)); they
    # are never handed to a chain kernel
    good = wi.config4(k=2, d=512, m=40, base_steps=10, mean_nnz=9.0, max_nnz=20).to("cuda")
    with P.Context(2, 512) as ctx:
        ctx.validate_csr(good.row_ptr, good.col_idx)
        ctx.check()
        nnz = int(good.col_idx.numel())
        row7 = slice(int(good.row_ptr[7]), int(good.row_ptr[8]))
        assert row7.stop - row7.start >= 2
        cases = []
        bad = good.col_idx.clone(); bad[row7.start] = 512            # column == d
        cases.append((good.row_ptr, bad, "detail 7"))
        bad = good.col_idx.clone(); bad[row7.start + 1] = -3          # negative column
        cases.append((good.row_ptr, bad, "detail 7"))
        bad = good.col_idx.clone(); bad[row7.start + 1] = bad[row7.start]   # a column twice in a row
        cases.append((good.row_ptr, bad, "detail 7"))
        rp = good.row_ptr.clone(); rp[0] = -1                         # row 0 starts before the arrays
        cases.append((rp, good.col_idx, "detail 0"))
        rp = good.row_ptr.clone(); rp[-1] = nnz + 10                  # last row claims entries beyond the arrays
        cases.append((rp, good.col_idx, f"detail {rp.numel() - 2}"))
        for rp_, ci_, where in cases:
            ctx.validate_csr(rp_, ci_)
            with pytest.raises(P.WpsgdError) as e:
                ctx.check()
            assert e.value.status_name == "CUDA" and where in str(e.value), str(e.value)
        ctx.validate_csr(good.row_ptr, good.col_idx)  # the context is clean again
        ctx.check()


def test_csr_equals_dense_kernels_on_densified_rows(P):
    wl = wi.config4(k=4, d=1024, m=128, base_steps=300, mean_nnz=20.0)
    wl.loss = LOGISTIC
    v_s, W_s, _, _ = gpu_solve(P, wl)
    v_d, W_d, _, _ = gpu_solve(P, wi.densify(wl))
    assert rel_l2(v_s, v_d) <= 1e-4


# ---- argument checking ----------------------------------------------------------------------------------------
def test_errors_are_reported_not_thrown_from_c(P):
    wl = wi.config1(k=2, d=64, m=16, n_steps=(5, 5)).to("cuda")
    with P.Context(2, 64) as ctx:
        with pytest.raises(P.WpsgdError) as e:
            ctx.combine()
        assert e.value.status_name == "STATE"
        with pytest.raises(P.WpsgdError) as e:
            ctx.get_models()
        assert e.value.status_name == "STATE"
        bad = [dict(n_steps=np.array([5, -1])), dict(shard_off=np.array([0, 16, 8])), dict(eta0=float("nan")),
               dict(lam=-1.0), dict(eta0=10.0, lam=0.2), dict(loss=9), dict(sched=5),
               dict(shard_off=np.array([0, 0, 32]), n_steps=np.array([3, 3]))]
        for kw in bad:
            args = dict(shard_off=wl.shard_off, n_steps=wl.n_steps, eta0=wl.eta0, sched=wl.sched, lam=wl.lam,
                        loss=wl.loss)
            args.update(kw)
            with pytest.raises(P.WpsgdError) as e:
                ctx.run(wl.X, wl.y, args["shard_off"], args["n_steps"], args["eta0"], args["sched"], args["lam"],
                        args["loss"], 0)
            assert e.value.status_name == "INVALID_ARG", kw
        with pytest.raises(P.WpsgdError):
            ctx.set_option("no_such_option", 1)
        with pytest.raises(P.WpsgdError):
            ctx.sample_indices(0, 0, 0, 0, 4)
        ctx.run_workload(wl)  # the context is still usable afterwards
        ctx.combine()
        ctx.check()
        assert ctx.launch_count() >= 3


# ---- shapes at the edges of the launch configurations ---------------------------------------------------------------
def test_many_nodes_with_few_steps(P):
    k, d, m = 3000, 64, 4
    g = torch.Generator().manual_seed(11)
    X = torch.randn(k * m, d, generator=g) / 8
    y = torch.sign(torch.randn(k * m, generator=g))
    n = (np.arange(k) % 7).astype(np.int64)  # 0..6 steps, many idle nodes, ragged last CTA
    wl = wi.Workload("many", k, d, np.arange(k + 1, dtype=np.int64) * m, n, 0.05, 0, 0.01, LOGISTIC, 5, y, X=X)
    assert_parity(P, wl)
    assert_parity(P, wl, {"dense_variant": 3})


@pytest.mark.parametrize("d", [1, 2, 3, 5])
def test_tiny_feature_counts(P, d):
    g = torch.Generator().manual_seed(d)
    k, m = 3, 20
    X = torch.randn(k * m, d, generator=g)
    y = torch.sign(torch.randn(k * m, generator=g))
    wl = wi.Workload("tiny", k, d, np.arange(k + 1, dtype=np.int64) * m, np.array([60, 1, 33]), 0.05, 0, 0.01, LOGISTIC, 3,
                     y, X=X)
    assert_parity(P, wl)


def test_one_long_chain(P):
    wl = wi.config2(k=1, d=256, m=512, base_steps=60000)
    assert_parity(P, wl)


def test_csr_rows_without_nonzeros_and_single_nonzero(P):
    # hand-built CSR: rows 0 and 3 are empty, row 1 has one nonzero, row 2 three
    rp = torch.tensor([0, 0, 1, 4, 4, 6], dtype=torch.int64)
    ci = torch.tensor([5, 0, 3, 7, 1, 6], dtype=torch.int32)
    va = torch.tensor([2.0, 0.5, -1.0, 0.25, 1.5, -0.75])
    y = torch.tensor([1.0, -1.0, 1.0, -1.0, 1.0])
    wl = wi.Workload("gaps", 1, 8, np.array([0, 5]), np.array([200]), 0.1, 1, 0.05, LOGISTIC, 2, y, row_ptr=rp, col_idx=ci,
                     val=va, w0=torch.full((8,), 0.3))
    assert_parity(P, wl)


# ---- CSR kernel: groups of 8 steps, forms by row length, rows at the edges of the chunks ---------------------------------
@pytest.mark.parametrize("lengths", [(1, 4, 5, 16), (16, 17, 31, 32), (33, 48, 63, 64), (65, 96, 97, 200), (0, 0, 1, 128)])
@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
def test_csr_group_forms(P, lengths, loss):
    # 16, 32 and 64 nonzeros are the limits of the compiled forms; step counts leave groups of 1, 7 and 8
    d = 1024
    rp, ci, va, y = _rows_with_given_lengths(list(lengths) * 3, d, 5)
    wl = wi.Workload("forms", 3, d, np.array([0, 4, 8, 12]), np.array([135, 96, 49]), 0.2, 1, 0.01, loss, 5, y, row_ptr=rp,
                     col_idx=ci, val=va, w0=torch.full((d,), 0.01))
    assert_parity(P, wl, {"sparse_variant": 2})


@pytest.mark.parametrize("d, lengths", [(32, (32,)), (34, (32, 31)), (33, (1, 32, 0, 7)), (2048, (10,)), (48, (20, 21)), (40, (5, 6, 10))])
@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
def test_csr_short_form_of_a_block(P, d, lengths, loss):
    # rows of at most 32 nonzeros, blocks of at most 640: every column shared by all rows of a group (d = 32), more shared
    # columns than lanes, hardly any (d = 2048); blocks on both sides of 640 follow one another where the rows differ
    rp, ci, va, y = _rows_with_given_lengths(list(lengths) * (24 // len(lengths)), d, 7)
    n = len(rp) - 1
    steps = np.array([203, 64, 17])
    wl = wi.Workload("short", 3, d, np.array([0, n // 3, 2 * (n // 3), n]), steps, 0.1, 1, 0.01, loss, 5, y, row_ptr=rp,
                     col_idx=ci, val=va, w0=torch.full((d,), 0.01))
    assert_parity(P, wl, {"sparse_variant": 2})


@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
def test_csr_chains_of_both_bodies_in_one_run(P, loss):
    # shards of 10 nonzeros per row on average (the limit of the body with the short form), just above, and far above; the
    # first also holds rows that fit no short block; the last shard is a single row without nonzeros
    d = 3000
    shards = [[3, 4, 5, 2, 40, 6, 20, 0], [10, 11, 9, 11, 10, 10, 10, 10], [40, 64, 33, 7], [0]]
    assert sum(shards[0]) == 10 * len(shards[0]) and sum(shards[1]) == 81
    rp, ci, va, y = _rows_with_given_lengths([n for s in shards for n in s], d, 9)
    off = np.concatenate([[0], np.cumsum([len(s) for s in shards])])
    wl = wi.Workload("bodies", 4, d, off, np.array([230, 230, 150, 20]), 0.1, 1, 0.01, loss, 5, y, row_ptr=rp, col_idx=ci, val=va,
                     w0=torch.full((d,), 0.01))
    assert_parity(P, wl, {"sparse_variant": 2})


@pytest.mark.parametrize("loss", [HINGE, LOGISTIC, SQUARED])
def test_csr_long_rows_one_step_at_a_time(P, loss):
    # blocks with more than 64 nonzeros per step (65; rows at the edges of the 128 that wait in registers; 2048, the most a block
    # takes; 2049 and 2560, which run on global memory), blocks just below, both kinds in turn, and long rows in a shard of
    # few nonzeros on average
    d = 6000
    shards = [[65, 65, 64, 66, 127, 128, 129, 256, 257], [2048, 65, 2049, 700, 2560, 513], [64, 63, 64, 65, 64, 64],
              [70, 300] + [2] * 60, [40, 40, 40, 400, 40, 40, 40, 40]]
    rp, ci, va, y = _rows_with_given_lengths([n for s in shards for n in s], d, 13)
    off = np.concatenate([[0], np.cumsum([len(s) for s in shards])])
    wl = wi.Workload("apart", 5, d, off, np.array([133, 60, 101, 400, 200]), 0.1, 1, 0.01, loss, 5, y, row_ptr=rp, col_idx=ci, val=va,
                     w0=torch.full((d,), 0.01))
    assert_parity(P, wl, {"sparse_variant": 2})


def test_csr_hinge_decisions_at_the_threshold(P):
    # two rows of the same columns with values chosen so that margins come within rounding of 1: the decisions have to be
    # those of one step at a time, as in the direct kernel (bit for bit the same models but for the fp64 scale's last bits)
    d, n = 64, 400
    g = torch.Generator().manual_seed(2)
    lengths = [8] * 40
    rp, ci, va, y = _rows_with_given_lengths(lengths, d, 3)
    va = (va * (1.0 + 1e-6 * torch.randn(va.shape, generator=g))).contiguous()
    wl = wi.Workload("ties", 2, d, np.array([0, 20, 40]), np.array([n, n // 2]), 0.25, 0, 0.0, HINGE, 5, y, row_ptr=rp, col_idx=ci, val=va)
    _, W2, _, _ = gpu_solve(P, wl, {"sparse_variant": 2})
    _, W1, _, _ = gpu_solve(P, wl, {"sparse_variant": 1})
    for j in range(2):
        assert rel_l2(W2[j], W1[j]) <= 1e-6
